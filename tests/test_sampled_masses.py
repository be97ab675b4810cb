"""Stochastic acceptance at vocabularies around the runs of 8192 logits whose masses are computed ahead of the walk, one and several runs,
rows that take vector loads and rows that do not, against the oracle's rule with the same uniforms."""
import numpy as np
import pytest

import parity
from paper_2503_01840_b200 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("temperature", [1.0, 3.0])
@pytest.mark.parametrize("vocab", [257, 8191, 8192, 8193, 24580])
def test_sampled_steps_by_vocabulary(vocab, temperature):
    """At temperature 3 the drawn token comes from anywhere in the row."""
    cfg = synth.C1.replace(name=f"V{vocab}", vocab=vocab, draft_vocab=200, batch=2, prompt_len=20)
    tw, dw = synth.make_target_weights(cfg), synth.make_draft_weights(cfg)
    rng = np.random.default_rng(vocab)
    prompts = [rng.integers(0, vocab, 20 + b).astype(np.int32) for b in range(2)]
    st, _ = parity.run_trajectory(cfg, tw, dw, prompts, n_steps=6, tol=1e-4, tap_tol=None, sampling=(temperature, 5))
    assert st.steps == 6 and st.verify_compared == 12 and st.passes == 12 * cfg.tree_depth, st


def test_more_verify_rows_than_a_grid_has_second_indexes():
    """1100 sequences of 60 verify rows: the first and the last sequences give what they give in a batch of their own."""
    from paper_2503_01840_b200 import binding as sb
    cfg = synth.ModelCfg("R", "fp32", 1, 32, 2, 1, 16, 64, 64, 48, (0, 0, 0), 1e4, tree_depth=2, tree_topk=8, tree_nodes=60, seed=9)
    tw, dw = synth.make_target_weights(cfg, device="cuda"), synth.make_draft_weights(cfg, device="cuda")
    B, steps = 1100, 3
    rng = np.random.default_rng(0)
    prompts = [rng.integers(0, cfg.vocab, 5).astype(np.int32) for _ in range(B)]
    u = rng.random((steps, B, 2 * cfg.tree_nodes), dtype=np.float32)
    picked = [0, 1, B - 2, B - 1]
    got = []
    for which in (range(B), picked):
        dec = sb.SpecDecoder(cfg.replace(batch=len(which)), tw, dw, batch=len(which), max_ctx=96)
        first = dec.prefill([prompts[b] for b in which], 16)
        out = [dec.step_sampled(1.0, u[i, list(which)]) for i in range(steps)]
        at = [list(which).index(b) for b in picked]
        got.append([first[at].tolist()] + [[o[b].tolist() for b in at] for o in out])
        dec.close()
    assert got[0] == got[1]
