"""The fp32 model's schedule with norms, RoPE, cache writes and activations on the GEMMs: every form of those kernels (4, 8, 16
rows), steps whose passes have more rows than they take, head dimensions and feature counts off the warps' shares, padding rows,
taps, against the CPU oracle; the rows they are taken for; weights off a 16-byte boundary stay on the plain schedule and agree with it."""
import numpy as np
import pytest

import parity
from paper_2503_01840_b200 import binding as sb
from paper_2503_01840_b200 import synth

pytestmark = pytest.mark.gpu

BASE = synth.ModelCfg("F", "fp32", 3, 72, 3, 1, 48, 200, 131, 77, (0, 1, 2), 5e5, tree_depth=3, tree_topk=2, tree_nodes=7, seed=23)


@pytest.mark.parametrize("kw,batch", [
    (dict(), 1),                                                       # 4, 2 and 7 rows
    (dict(tree_topk=4, tree_nodes=16), 1),                             # 16 rows
    (dict(n_heads=4, n_kv_heads=2, head_dim=16, ffn=136, tree_topk=5, tree_nodes=29), 1),     # 4 and 5 rows, 29 on the plain schedule
    (dict(tree_depth=2, tree_topk=3, tree_nodes=11), 3),               # 9 and 9 rows, 33 on the plain schedule
    (dict(hidden=256, n_heads=2, n_kv_heads=2, head_dim=80, ffn=688, tree_depth=4, tree_nodes=12), 5),   # 10 rows, 25 and 60 on the plain schedule
], ids=str)
def test_fp32_schedule_vs_oracle(kw, batch):
    cfg = BASE.replace(batch=batch, prompt_lo=5, prompt_hi=70, prompt_len=37, **kw)
    tw, dw = synth.make_target_weights(cfg), synth.make_draft_weights(cfg)
    prompts = [p.numpy() for p in synth.make_prompts(cfg)]
    st, _ = parity.run_trajectory(cfg, tw, dw, prompts, n_steps=4, tol=1e-4)
    assert st.passes == 4 * cfg.tree_depth * batch and st.verify_compared == 4 * batch, st


@pytest.mark.parametrize("hidden,most", [(64, 16), (256, 16), (264, 8), (1024, 8)])
def test_fp32_rows_the_schedule_is_taken_for(hidden, most):
    """Up to 16 rows at short contractions, up to 8 at others: seen by the launches of a step whose draft passes have few rows."""
    def launches(rows):
        cfg = BASE.replace(hidden=hidden, tree_depth=6, tree_topk=4, tree_nodes=rows)
        tw, dw = synth.make_target_weights(cfg, device="cuda"), synth.make_draft_weights(cfg, device="cuda")
        dec = sb.SpecDecoder(cfg, tw, dw, batch=1, max_ctx=64)
        dec.prefill([np.arange(20, dtype=np.int32)], 10)
        dec.step()
        n = dec.launches_per_step()
        dec.close()
        return n

    few = launches(3)
    assert launches(most) == few
    assert launches(most + 1) > few


def test_fp32_unaligned_norm_weights():
    """Norm gains off a 16-byte boundary take the plain schedule; both are fp32 sums of the same products."""
    import torch
    cfg = BASE.replace(hidden=256, n_heads=4, n_kv_heads=2, head_dim=64, tree_nodes=12)
    tw, dw = synth.make_target_weights(cfg, device="cuda"), synth.make_draft_weights(cfg, device="cuda")

    def shifted(t):
        buf = torch.empty(t.numel() + 1, device="cuda")
        buf[1:].copy_(t.view(-1))
        return buf[1:].view(t.shape)

    def off_grid(w):
        return {k: [off_grid(x) for x in v] if isinstance(v, list) else shifted(v) if "norm" in k else v for k, v in w.items()}

    prompt, hidden = [np.arange(40, dtype=np.int32) % cfg.vocab], []
    for t, d in ((tw, dw), (off_grid(tw), off_grid(dw))):
        dec = sb.SpecDecoder(cfg, t, d, batch=1, max_ctx=160)
        dec.prefill(prompt, 16)
        dec.step()
        hidden.append((dec.debug(sb.DBG_TREE_TOK), dec.debug(sb.DBG_NODE_HIDDEN)))
        dec.close()
    assert np.array_equal(hidden[0][0], hidden[1][0])
    a, b = hidden[0][1].astype(np.float64), hidden[1][1].astype(np.float64)
    assert np.abs(a - b).max() <= 2e-5 * np.sqrt((b * b).mean())         # sums of up to 400 products, three layers deep


def test_fp32_heads_off_the_schedule():
    """LM heads off a 16-byte boundary run behind a closing norm of their own, which takes the residual stream from where the last
    layer left it (a copy inside the captured step)."""
    import torch
    cfg = BASE.replace(hidden=256, n_heads=4, n_kv_heads=2, head_dim=64, tree_nodes=12)
    tw, dw = synth.make_target_weights(cfg, device="cuda"), synth.make_draft_weights(cfg, device="cuda")

    def shifted(t):
        buf = torch.empty(t.numel() + 1, device="cuda")
        buf[1:].copy_(t.view(-1))
        return buf[1:].view(t.shape)

    tws, dws = dict(tw, lm_head=shifted(tw["lm_head"])), dict(dw, lm_head=shifted(dw["lm_head"]))
    prompt, seen = [np.arange(40, dtype=np.int32) % cfg.vocab], []
    for t, d, flags in ((tw, dw, 0), (tws, dws, 0), (tws, dws, sb.FLAG_NO_GRAPH)):
        dec = sb.SpecDecoder(cfg, t, d, batch=1, max_ctx=160, flags=flags)
        dec.prefill(prompt, 16)
        ids = np.concatenate([dec.step()[0] for _ in range(3)])
        seen.append((ids, dec.debug(sb.DBG_TREE_TOK), dec.debug(sb.DBG_NODE_HIDDEN), dec.debug(sb.DBG_TARGET_LOGITS)))
        dec.close()
    assert all(np.array_equal(x, y) for x, y in zip(seen[1], seen[2]))
    for a, b in zip(seen[0][:2], seen[1][:2]):
        assert np.array_equal(a, b)
    for a, b in zip(seen[0][2:], seen[1][2:]):
        a, b = a.astype(np.float64), b.astype(np.float64)
        assert np.abs(a - b).max() <= 2e-5 * np.sqrt((b * b).mean())     # sums of up to 400 products, three layers deep


@pytest.mark.parametrize("rows", [1, 4, 5, 16, 17, 33])
@pytest.mark.parametrize("O,I", [(33, 380), (33, 384), (250, 388), (2, 516), (70, 1028), (1184, 640), (4744, 512)])
def test_fp32_gemm_contraction_over_warps(rows, O, I):
    """Contractions around the length from which a block's warps share them, remainders of the 512 elements they take at a time,
    and feature counts on both sides of the blocks that are resident together."""
    _gemm_vs_fp64(rows, O, I)


@pytest.mark.parametrize("rows,O,I", [(4, 3552, 388), (4, 3560, 1020), (4, 3560, 1024), (4, 7112, 1532), (4, 7112, 1536), (7, 2372, 508), (7, 2372, 512),
                                      (13, 890, 388), (13, 1778, 508), (13, 1778, 512), (30, 592, 388), (30, 594, 508), (30, 594, 512), (30, 1186, 1020),
                                      (30, 1186, 1024), (30, 1778, 1028)])
def test_fp32_gemm_blocks_around_waves(rows, O, I):
    """Feature counts on both sides of one, two and three waves of each form, contractions on both sides of where they are taken."""
    _gemm_vs_fp64(rows, O, I)


def _gemm_vs_fp64(rows, O, I):
    import torch
    g = torch.Generator().manual_seed(rows + O + I)
    x, w = torch.randn(rows, I, generator=g), torch.randn(O, I, generator=g)
    out = sb.gemm(x.cuda(), w.cuda(), impl=1).cpu().double().numpy()
    xd, wd = x.double().numpy(), w.double().numpy()
    bound = 2.0 ** -23 * (8 + I / 32) * (np.abs(xd) @ np.abs(wd).T)     # lane sums of up to I / 32 products, then eight exchanges
    assert (np.abs(out - xd @ wd.T) <= bound + 1e-30).all()
