"""Host rules of the kernels that no entry point shows, asked of the built library by a small program (no GPU: nothing is launched)."""
import os
import subprocess

import pytest

from paper_2503_01840_b200 import binding as sb
from paper_2503_01840_b200 import build

ASK = r"""
#include <cstdio>
#include <cstdlib>
#include "attn_fast.cuh"
#include "gemm_fused.cuh"
#include "state.cuh"
using namespace spec;
int main(int n, char **v) {                     // epilogue, rows, split, stages; or rows, rows per sequence, context, tail, grows (32 heads, 8 KV heads)
  if (v[1][0] == 'a') { printf("%d", attn_ref_reads_ahead(atoi(v[2]), atoi(v[3]), atoi(v[4]), atoi(v[5])) ? 1 : 0); return 0; }      // "ahead", rows, heads, head size, keys
  if (v[1][0] == 'v') { printf("%d", accept_sampled_takes(atoi(v[2])) ? accept_mass_chunks(atoi(v[2])) : -accept_mass_chunks(atoi(v[2]))); return 0; }      // "vocabulary", ids
  if (n == 7) { printf("%d", attn_fast_plan(atoi(v[1]), 32, 8, 128, atoi(v[2]), atoi(v[3]), atoi(v[4]), atoi(v[5]) != 0, atoi(v[6]) != 0) >> 1); return 0; }      // ... and TMA
  if (n == 6) { printf("%d", attn_fast_plan(atoi(v[1]), 32, 8, 128, atoi(v[2]), atoi(v[3]), atoi(v[4]), atoi(v[5]) != 0) >> 1); return 0; }
  static char mem[64];
  FusedGemmArgs a;
  const FusedEpi epi = (FusedEpi)atoi(v[1]);
  a.x = (const bf16 *)(((uintptr_t)mem + 15) & ~(uintptr_t)15);
  a.w[0] = a.w[1] = a.x;
  a.O[0] = a.O[1] = 512; a.I = 512; a.nw = epi == EPI_SWIGLU ? 2 : 1;
  a.rows = atoi(v[2]); a.split = atoi(v[3]); a.stages = atoi(v[4]);
  printf("%d", fused_gemm_supported(epi, a) ? 1 : 0);
}
"""


@pytest.fixture(scope="module")
def ask(tmp_path_factory):
    d = tmp_path_factory.mktemp("rules")
    src, exe = d / "ask.cu", d / "ask"
    src.write_text(ASK)
    lib = sb.library_path()
    sb.lib()
    subprocess.run([build.NVCC, "-std=c++17", "-gencode", "arch=compute_100a,code=sm_100a", "-I", build.CSRC, str(src), lib, "-o", str(exe),
                    "-Xlinker", "-rpath", "-Xlinker", os.path.dirname(lib)], check=True, capture_output=True)
    return lambda *args: int(subprocess.run([str(exe), *map(str, args)], check=True, capture_output=True).stdout)


F32, SWIGLU = 0, 3


@pytest.mark.parametrize("rows,split,stages,taken", [
    (128, 0, 0, 1), (128, 2, 0, 1), (128, 0, 3, 1), (256, 0, 0, 1), (129, 0, 0, 1),
    (129, 2, 0, 0), (129, 0, 3, 0), (256, 1, 0, 0), (256, 4, 4, 0),
])
def test_gate_up_plans_are_for_up_to_128_rows(ask, rows, split, stages, taken):
    """A forced K split or ring depth exists for gate/up up to 128 rows only: beyond, the tile kernel would read 256-row activation
    boxes into stages of 128 rows."""
    assert ask(SWIGLU, rows, split, stages) == taken
    assert ask(F32, rows, split, stages) == 1


@pytest.mark.parametrize("rows,rps,ctx,tail,now,growing", [
    (1, 1, 700, 64, 12, 13),        # 18 splits would fit: as many as key tiles
    (1, 1, 10, 1, 1, 2),
    (60, 60, 10, 60, 2, 3),
    (60, 60, 512, 60, 9, 5),        # 9 fit: 9 tiles, one each; 10 tiles, two each
    (60, 60, 580, 60, 5, 6),        # 10 tiles; 11
    (256, 4, 2000, 4, 1, 1),
])
def test_key_splits_of_a_launch_and_of_a_step_that_grows(ask, rows, rps, ctx, tail, now, growing):
    """No split without a key tile where the hint is the length; a captured step has one tile to grow by."""
    assert ask(rows, rps, ctx, tail, 0) == now
    assert ask(rows, rps, ctx, tail, 1) == growing


@pytest.mark.parametrize("rows,H,hd,keys,ahead", [
    (1, 4, 64, 100, 1), (148, 4, 64, 100, 1), (149, 4, 64, 100, 0), (240, 4, 64, 600, 0), (60, 32, 96, 2000, 0),
    (60, 32, 96, 14000, 0), (60, 32, 96, 14700, 1),                 # four or three CTAs of the small form in an SM's 228 KB
    (1, 1, 64, 58028, 1), (1, 1, 64, 58033, 0),                     # 227 KB
    (262144, 64, 128, 100, 0),
])
def test_plain_attention_reads_ahead_in_two_waves(ask, rows, H, hd, keys, ahead):
    assert ask("ahead", rows, H, hd, keys) == ahead


@pytest.mark.parametrize("vocab,chunks", [(2, 1), (8192, 1), (8193, 2), (128256, 16), (1 << 26, 8192), ((1 << 26) + 1, -8193), (2 ** 31 - 1, -262144)])
def test_vocabularies_of_the_stochastic_acceptance(ask, vocab, chunks):
    """Runs of 8192 ids; one CTA's shared memory holds the masses of 8192 runs, and a larger vocabulary is refused."""
    assert ask("vocabulary", vocab) == chunks


@pytest.mark.parametrize("seqs,ctx,grows,one_cta,two_ctas", [
    (1, 700, 0, 11, 11), (2, 700, 0, 6, 6),                          # 11 tiles: one wave of one CTA an SM already gives most of them a tile each
    (2, 2000, 0, 8, 16), (4, 700, 0, 4, 4),                          # 32 tiles, two each; 11 tiles in 4 or in 5 splits are three each
    (6, 700, 0, 3, 4), (6, 2000, 0, 3, 6), (6, 60, 0, 1, 1),         # no split for less than two tiles
    (12, 700, 0, 1, 3), (12, 700, 1, 1, 3), (18, 700, 0, 1, 2), (18, 120, 1, 1, 1),
    (36, 700, 0, 1, 1), (37, 700, 0, 1, 1), (64, 2000, 1, 1, 1),
])
def test_key_splits_of_chains(ask, seqs, ctx, grows, one_cta, two_ctas):
    """Up to 16 query rows per KV head (four rows, four heads a group): the key-parallel kernel, two of whose CTAs an SM holds, is split for 296
    CTAs as long as each keeps two tiles; without TMA another kernel takes the launch, one CTA an SM."""
    assert ask(4 * seqs, 4, ctx, 4, grows, 0) == one_cta
    assert ask(4 * seqs, 4, ctx, 4, grows, 1) == ask(4 * seqs, 4, ctx, 4, grows) == two_ctas


@pytest.mark.parametrize("seqs,ctx", [(2, 700), (6, 2000), (18, 700)])
def test_key_splits_of_trees_do_not_depend_on_tma(ask, seqs, ctx):
    """More than 16 query rows: one CTA an SM either way."""
    assert ask(20 * seqs, 20, ctx, 20, 0, 0) == ask(20 * seqs, 20, ctx, 20, 0, 1)
