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
