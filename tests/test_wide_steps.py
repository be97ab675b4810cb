"""Steps whose passes have 129 to 256 rows (the row-major GEMM kernel, split over K slices or not), and batches whose pass
over the pending entries goes on with one row per sequence, against the CPU oracle."""
import pytest

import parity
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
