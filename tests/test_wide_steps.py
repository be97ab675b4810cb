"""Steps whose passes have 129 to 256 rows (the row-major GEMM kernel, split over K slices or not), and batches whose pass
over the pending entries goes on with one row per sequence, against the CPU oracle."""
import numpy as np
import pytest
import torch

import parity
from paper_2503_01840_b200 import binding as sb
from paper_2503_01840_b200 import synth

pytestmark = pytest.mark.gpu

W4 = synth.ModelCfg("W4", "bf16", 2, 512, 8, 2, 128, 1408, 2050, 1024, (0, 1, 1), 5e5, tree_depth=4, tree_topk=5, tree_nodes=24, seed=41)
# a contraction long enough for several K slices, feature counts off the tile grid
L4 = W4.replace(name="L4", hidden=1160, ffn=2056, n_heads=4)


@pytest.mark.parametrize("cfg,batch,nodes,sampled", [
    (W4, 3, 43, False),      # 129 rows: one row in the second half of the row tile
    (W4, 4, 48, True),       # 192: the last gate/up launch of the weight-streaming kernel, logits written out
    (W4, 5, 39, False),      # 195: the first of the row-major kernel; a vocabulary of 16 tiles and two features
    (W4, 4, 64, True), (L4, 4, 64, False), (L4, 3, 45, True),
], ids=lambda v: getattr(v, "name", str(v)))
def test_wide_verify_passes_vs_oracle(cfg, batch, nodes, sampled):
    cfg = cfg.replace(name=f"{cfg.name}-b{batch}n{nodes}", batch=batch, tree_nodes=nodes, prompt_lo=20, prompt_hi=90)
    tw, dw = synth.make_target_weights(cfg), synth.make_draft_weights(cfg)
    prompts = [p.numpy() for p in synth.make_prompts(cfg)]
    st, _ = parity.run_trajectory(cfg, tw, dw, prompts, n_steps=3, tol=2e-2, tap_tol=3e-2, sampling=(0.8, 7) if sampled else None)
    assert st.passes == 3 * cfg.tree_depth * batch and st.verify_compared == 3 * batch, st


@pytest.mark.parametrize("batch,depth", [(4, 4), (17, 3), (40, 3), (64, 3)])
def test_pending_pass_goes_on_with_one_row_per_sequence(batch, depth):
    """20 -> 4, 68 -> 17, 160 -> 40 and 256 -> 64 rows after the attention of the first draft pass."""
    cfg = W4.replace(name=f"chain-b{batch}", batch=batch, tree_depth=depth, tree_topk=1, tree_nodes=depth + 1, prompt_lo=5, prompt_hi=40)
    tw, dw = synth.make_target_weights(cfg), synth.make_draft_weights(cfg)
    prompts = [p.numpy() for p in synth.make_prompts(cfg)]
    st, _ = parity.run_trajectory(cfg, tw, dw, prompts, n_steps=3, tol=2e-2, tap_tol=3e-2)
    assert st.passes == 3 * depth * batch and st.verify_compared == 3 * batch, st


@pytest.mark.parametrize("batch,draft_vocab", [(9, 1003), (9, 1008), (16, 1002)])
def test_unfused_draft_logits_of_wide_passes(batch, draft_vocab):
    """Sixteen candidates per node: the draft logits are written out (144 and 256 rows), for vocabularies that are and are
    not a multiple of eight."""
    cfg = W4.replace(name=f"k16-b{batch}-v{draft_vocab}", batch=batch, draft_vocab=draft_vocab, tree_depth=2, tree_topk=16, tree_nodes=16,
                     prompt_lo=5, prompt_hi=40)
    tw, dw = synth.make_target_weights(cfg), synth.make_draft_weights(cfg)
    prompts = [p.numpy() for p in synth.make_prompts(cfg)]
    st, _ = parity.run_trajectory(cfg, tw, dw, prompts, n_steps=2, tol=2e-2, tap_tol=3e-2)
    assert st.passes == 2 * 2 * batch and st.verify_compared == 2 * batch, st


@pytest.mark.parametrize("kernel,hidden,prompt", [(1, 4096, 1300), (2, 512, 150), (3, 512, 150)])
def test_row_major_wait_that_runs_out_is_reported(kernel, hidden, prompt):
    """One CTA of each row-major kernel never receives its first activation tile (test hook): its bounded waits run out, the
    CTAs of its cluster wind down, and the prefill returns the site of the wait.  A fresh decoder works afterwards."""
    cfg = W4.replace(name="wait", hidden=hidden, n_heads=hidden // 128, n_kv_heads=max(2, hidden // 512), ffn=1024 if hidden == 4096 else 1408,
                     batch=1 if hidden == 4096 else 4, tree_nodes=64)
    tw, dw = synth.make_target_weights(cfg, device="cuda"), synth.make_draft_weights(cfg, device="cuda")
    rng = np.random.default_rng(4)
    prompts = [rng.integers(0, cfg.vocab, prompt).astype(np.int32) for _ in range(cfg.batch)]
    seen = []
    for hook in (0, kernel, 0):
        dec = sb.SpecDecoder(cfg, tw, dw, batch=cfg.batch, max_ctx=prompt + 200)
        sb.lib().spec_debug_wide_gemm(hook)
        try:
            if not hook:
                seen.append([dec.prefill(prompts, 16), *dec.step()])
                continue
            with pytest.raises(sb.SpecError) as e:
                dec.prefill(prompts, 16)
            assert e.value.code == -7 and f"site {23 + kernel}" in str(e.value), str(e.value)
        finally:
            sb.lib().spec_debug_wide_gemm(0)
            dec.close()
    assert all(np.array_equal(a, b) for a, b in zip(*seen))


@pytest.mark.parametrize("topk", [5, 16])
def test_draft_logits_that_are_not_numbers(topk):
    """A draft whose logits are all NaN gives some tree of valid tokens (fused and separate expansion kernels), and the steps
    emit what plain decoding emits."""
    cfg = W4.replace(name="nan", batch=2, tree_depth=3, tree_topk=topk)
    tw, dw = synth.make_target_weights(cfg, device="cuda"), synth.make_draft_weights(cfg, device="cuda")
    dw["lm_head"] = torch.full_like(dw["lm_head"], float("nan"))
    prompts = [np.arange(30, dtype=np.int32), np.arange(7, 40, dtype=np.int32)]
    spec, plain = (sb.SpecDecoder(cfg, tw, dw, batch=2, max_ctx=300) for _ in range(2))
    assert np.array_equal(spec.prefill(prompts, 32), plain.prefill(prompts, 32))
    out = [np.concatenate(x) for x in zip(spec.step(), spec.step())]
    ref = np.stack([plain.plain_step() for _ in range(max(map(len, out)))], 1)
    # one decision can be a near-tie that another order of sums turns: the first token of each sequence is compared
    assert all(o[0] == r[0] and ((0 <= o) & (o < cfg.vocab)).all() for o, r in zip(out, ref))
    spec.close()
    plain.close()


def _off_grid(weights):
    """The same weights with every norm vector one element (two bytes) behind an 8-byte boundary."""
    def move(t):
        buf = torch.empty(t.numel() + 4, dtype=t.dtype, device=t.device)
        buf[1 : 1 + t.numel()] = t
        return buf[1 : 1 + t.numel()]

    out = {n: move(t) if n.endswith("norm") else t for n, t in weights.items()}
    if "layers" in out:
        out["layers"] = [_off_grid(layer) for layer in out["layers"]]
    return out


@pytest.mark.parametrize("cfg,batch,prompt", [
    (W4, 4, 150),                                                                       # 256-row steps and a prefill, split over K
    (W4.replace(name="W4-wide", hidden=4096, n_heads=32, n_kv_heads=8, ffn=1024), 1, 1300),   # 96 tiles: the persistent kernel
], ids=lambda v: getattr(v, "name", str(v)))
def test_norm_weights_need_no_alignment(cfg, batch, prompt):
    """Norm gains off an 8-byte boundary give the bits that aligned ones give."""
    cfg = cfg.replace(batch=batch, tree_nodes=64)
    tw, dw = synth.make_target_weights(cfg, device="cuda"), synth.make_draft_weights(cfg, device="cuda")
    rng = np.random.default_rng(3)
    prompts = [rng.integers(0, cfg.vocab, prompt).astype(np.int32) for _ in range(batch)]
    seen = []
    for t, d in ((tw, dw), (_off_grid(tw), _off_grid(dw))):
        dec = sb.SpecDecoder(cfg, t, d, batch=batch, max_ctx=prompt + 200)
        got = [dec.prefill(prompts, 16)]
        got += [x for _ in range(2) for x in dec.step()]
        got += [dec.debug(sb.DBG_NODE_HIDDEN, b) for b in range(batch)] + list(dec.read_kv(0, -1, prompt - 2))
        seen.append(got)
        dec.close()
    assert all(np.array_equal(x, y) for x, y in zip(*seen)) and np.isfinite(seen[0][-1]).all()
