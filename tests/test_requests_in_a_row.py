"""Requests of different lengths and modes one after the other on one context: whatever a context keeps from one request to the
next (captured steps, staging buffers), each gives the bits that a context of its own gives."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,batch", [("fp32", 1), ("fp32", 2), ("bf16", 1), ("bf16", 3)])
def test_requests_in_a_row_equal_fresh_contexts(dtype, batch):
    _requests_in_a_row(dtype, batch, 0)


@pytest.mark.parametrize("flags", ["FLAG_REF_GEMM", "FLAG_REF_ATTN", "FLAG_NO_TMA_ATTN", "FLAG_NO_PDL"])
def test_requests_in_a_row_on_other_kernels(flags):
    from paper_2503_01840_b200 import binding as sb
    _requests_in_a_row("bf16", 2, getattr(sb, flags))


def _requests_in_a_row(dtype, batch, flags):
    from paper_2503_01840_b200 import binding as sb
    from paper_2503_01840_b200 import synth
    cfg = synth.ModelCfg("R", dtype, 2, 256, 4, 2, 64 if dtype == "fp32" else 128, 688, 2048, 1000, (0, 1, 1), 5e5, tree_depth=4, tree_topk=4, tree_nodes=20, seed=17).replace(batch=batch)
    tw, dw = synth.make_target_weights(cfg, device="cuda"), synth.make_draft_weights(cfg, device="cuda")
    rng = np.random.default_rng(5)
    # lengths on both sides of a change of the key split, repeated lengths, and the modes mixed
    requests = [(40, "greedy"), (44, "greedy"), (700, "greedy"), (700, "sampled"), (30, "plain"), (41, "greedy"), (700, "sampled"), (640, "greedy")]
    u = rng.random((batch, 2 * cfg.tree_nodes), dtype=np.float32)

    def serve(dec, n, mode):
        got = [dec.prefill([np.random.default_rng(n + b).integers(0, cfg.vocab, n + 3 * b).astype(np.int32) for b in range(batch)], 40)]
        for _ in range(3):
            got += [dec.plain_step()] if mode == "plain" else dec.step_sampled(0.8, u) if mode == "sampled" else dec.step()
        hidden = [] if mode == "plain" else [dec.debug(sb.DBG_NODE_HIDDEN, b) for b in range(batch)]      # (a plain pass has one row per sequence)
        return got + [dec.lengths()] + hidden

    one = sb.SpecDecoder(cfg, tw, dw, batch=batch, max_ctx=800, flags=flags)
    for n, mode in requests:
        fresh = sb.SpecDecoder(cfg, tw, dw, batch=batch, max_ctx=800, flags=flags)
        a, b = serve(one, n, mode), serve(fresh, n, mode)
        fresh.close()
        assert len(a) == len(b) and all(np.array_equal(x, y) for x, y in zip(a, b)), (n, mode)
    one.close()
