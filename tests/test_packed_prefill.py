"""The packed prefill (wide GEMM, causal tcgen05 attention) against the CPU oracle, at the edges of its tiles and passes."""
import numpy as np
import pytest

import parity
import pyoracle as po
from paper_2503_01840_b200 import binding as sb
from paper_2503_01840_b200 import synth

pytestmark = pytest.mark.gpu

# head_dim 128, four query heads per KV head; 3 layers of which none after the first two is tapped (P4), or all are (A4)
P4 = synth.ModelCfg("P4-gqa", "bf16", 3, 512, 8, 2, 128, 1408, 2048, 1024, (0, 1, 1), 5e5, tree_depth=2, tree_topk=4, tree_nodes=12, seed=31)
A4 = P4.replace(name="A4-all-tapped", fuse_layers=(0, 1, 2))
# one and three query heads per KV head (a CTA takes two blocks of positions instead of two heads), odd widths, page sizes
M1 = synth.ModelCfg("M1-mha", "bf16", 2, 520, 4, 4, 128, 1032, 2048, 1024, (0, 0, 1), 1e4, tree_depth=2, tree_topk=4, tree_nodes=12, seed=32)
G3 = P4.replace(name="G3-group3", n_heads=6, hidden=392, ffn=904, page_size=64)


@pytest.mark.parametrize("cfg,lens", [
    (P4, [1]), (P4, [2]), (P4, [128]), (P4, [256]), (P4, [257]), (P4, [513]),
    (A4, [129, 1, 300]),                                   # one pass, a prompt of one token among others
    (P4.replace(page_size=32), [255, 640, 66]),
    (P4, [4090, 40]),                                      # more rows than a pass holds: the second prompt starts in pass 1
    (P4, [30, 4200]),                                      # a prompt cut by a pass boundary off its block grid
    (M1, [130]), (M1, [257, 500, 3]), (M1, [260, 4100]), (G3, [383, 129]),
], ids=lambda v: v.name if hasattr(v, "name") else "-".join(map(str, v)))
def test_packed_prefill_vs_oracle(cfg, lens):
    """First tokens, the committed K/V of every layer (the draft's too) around every tile and block edge, and one step."""
    cfg = cfg.replace(batch=len(lens))
    tw, dw = synth.make_target_weights(cfg), synth.make_draft_weights(cfg)
    rng = np.random.default_rng(sum(lens))
    prompts = [rng.integers(0, cfg.vocab, n).astype(np.int32) for n in lens]
    st, _ = parity.run_trajectory(cfg, tw, dw, prompts, n_steps=1, tol=2e-2, tap_tol=3e-2, page_shuffle_seed=5, greedy_check=False)
    assert st.passes == cfg.tree_depth * len(lens) and st.verify_compared == len(lens), st
    dec = sb.SpecDecoder(cfg, parity.to_dev(tw), parity.to_dev(dw), batch=len(lens), max_ctx=max(lens) + 64, page_shuffle_seed=6)
    dec.prefill(prompts, 8)
    passes = dec.debug(sb.DBG_PREFILL_PASSES)
    assert passes.sum() == sum(lens) and (len(passes) > 1) == (sum(lens) > 4000), passes
    cuts = np.cumsum(passes)[:-1].tolist()
    for b, n in enumerate(lens):
        orc = po.Oracle(cfg, tw, dw, n + 64)
        orc.prefill(prompts[b])
        edges = {0, 1, 63, 64, 127, 128, 129, 255, 256, 257, n // 2, n - 3, n - 2, n - 1}
        edges |= {e - sum(lens[:b]) + d for e in cuts for d in (-1, 0, 1)}             # around every pass boundary
        for pos in sorted(e for e in edges if 0 <= e < n):
            for layer in range(cfg.n_layers):
                gk, gv = dec.read_kv(b, layer, pos)
                ok, ov = orc.target_kv(layer, pos)
                assert np.abs(gk - ok).max() < 8e-2 and np.abs(gv - ov).max() < 8e-2, (b, pos, layer)
            if pos < n - 1:
                gk, gv = dec.read_kv(b, -1, pos)
                ok, ov = orc.draft_kv(pos)
                assert np.abs(gk - ok).max() < 8e-2 and np.abs(gv - ov).max() < 8e-2, (b, pos, "draft")
    dec.close()
