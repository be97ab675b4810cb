"""Single kernels of a step, launched on inputs of a test's own: no entry point takes them.  A small library around their launchers
is compiled against the headers and linked to the built one."""
import ctypes as C
import functools
import os
import subprocess
import tempfile

import torch

from paper_2503_01840_b200 import binding as sb
from paper_2503_01840_b200 import build

SOURCE = r"""
#include "state.cuh"
using namespace spec;
extern "C" {
static int done() { return cudaGetLastError() == cudaSuccess && cudaDeviceSynchronize() == cudaSuccess ? 0 : -1; }
int mass_chunks(int V) { return accept_mass_chunks(V); }
// state: [5][B] n, n_prev, P, root, active; out: [3][B * (D + 1)] path, ids, pending, then [B] counts
int accept_sampled(const float *logits, int V, const float *u, float2 *mass, int32_t *tok, int32_t *parent, int32_t *nn, int32_t *state, int32_t *out, int B, int N, int D) {
  SeqState st = {};
  st.n = state; st.n_prev = state + B; st.P = state + 2 * B; st.root = state + 3 * B; st.active = state + 4 * B;
  TreeBufs tb = {};
  tb.N = N; tb.D = D; tb.Pmax = D + 1; tb.tok = tok; tb.parent = parent; tb.nn = nn;
  const int e = B * (D + 1);
  tb.path = out; tb.out_ids = out + e; tb.pend_tok = out + 2 * e; tb.out_cnt = out + 3 * e;
  const int n = launch_accept_sampled(st, tb, logits, V, u, mass, B, N, 0);
  return done() == 0 ? n : -1;
}
static RowMeta rows_of(int32_t *m, uint64_t *masks, int rows) {
  RowMeta r;
  r.seq = m; r.pos = m + rows; r.kvpos = m + 2 * rows; r.ctx = m + 3 * rows; r.tail_base = m + 4 * rows; r.tok = m + 5 * rows;
  r.mask_lo = masks; r.mask_hi = masks + rows;
  return r;
}
// pool: [3][B * (pool + 1)] tokens, parents, depths; tree: [4][B * N] tokens, parents, depths, pool indices; state: [2][B] n, active
int rerank(int32_t *pool_i, float *score, int32_t *state, int32_t *tree, float *tree_score, uint64_t *tree_mask, int32_t *nn, int32_t *meta, uint64_t *masks, int B, int pool, int N) {
  SeqState st = {};
  st.n = state; st.active = state + B;
  TreeBufs tb = {};
  const int pe = B * (pool + 1), ne = B * N;
  tb.pool = pool; tb.N = N; tb.pool_tok = pool_i; tb.pool_parent = pool_i + pe; tb.pool_depth = pool_i + 2 * pe; tb.pool_score = score;
  tb.tok = tree; tb.parent = tree + ne; tb.depth = tree + 2 * ne; tb.poolidx = tree + 3 * ne; tb.score = tree_score; tb.mask = tree_mask; tb.nn = nn;
  launch_rerank(st, tb, rows_of(meta, masks, ne), B, 0);
  return done();
}
int cand_pitch(int tiles) { return draft_tree_cand_ld(tiles); }
// state: [3][B] n, active, last_row; front: [B * D * K] frontier, [B * K] current frontier, [B * K] feature rows; top: [B * K * K] ids
int tree_step(int32_t *state, int32_t *pool_i, float *score, int32_t *front, int32_t *top, float *top_lp, int32_t *meta, uint64_t *masks, const int32_t *d2t, int pass,
              const float *cand_val, const int32_t *cand_idx, const float *cand_max, const float *cand_sum, int tiles, const float *x, const void *embed, void *cat, int k,
              const double *inv_freq, float2 *cs, int half, int B, int K, int D) {
  SeqState st = {};
  st.n = state; st.active = state + B; st.last_row = state + 2 * B;
  TreeBufs tb = {};
  tb.K = K; tb.D = D; tb.pool = K + (D - 1) * K * K;
  const int pe = B * (tb.pool + 1);
  tb.pool_tok = pool_i; tb.pool_parent = pool_i + pe; tb.pool_depth = pool_i + 2 * pe; tb.pool_score = score;
  tb.frontier = front; tb.front_cur = front + B * D * K; tb.feat_row = tb.front_cur + B * K; tb.tk_idx = top; tb.tk_lp = top_lp;
  const int rc = launch_draft_tree_step(st, tb, rows_of(meta, masks, B * K), d2t, pass, cand_val, cand_idx, cand_max, cand_sum, tiles, draft_tree_cand_ld(tiles), x,
                                        (const bf16 *)embed, (bf16 *)cat, k, inv_freq, cs, half, B, false, 0);
  return done() == 0 ? rc : -2;
}
}
"""


@functools.lru_cache(None)
def library():
    path = sb.library_path()
    sb.lib()
    with tempfile.TemporaryDirectory() as d:
        src, out = os.path.join(d, "step_kernels.cu"), os.path.join(d, "step_kernels.so")
        with open(src, "w") as f:
            f.write(SOURCE)
        subprocess.run([build.NVCC, *build.FLAGS, "-shared", "-I", build.CSRC, src, path, "-o", out, "-Xlinker", "-rpath", "-Xlinker", os.path.dirname(path)], check=True,
                       capture_output=True)
        return C.CDLL(out)


def call(name, *args):
    """Tensors by address, numbers as they are."""
    torch.cuda.synchronize()
    return getattr(library(), name)(*[None if a is None else C.c_void_p(a.data_ptr()) if isinstance(a, torch.Tensor) else C.c_int(a) for a in args])
