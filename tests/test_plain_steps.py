"""What spec_debug_read gives after a plain step: the step's one row of each sequence, not the rows of an earlier tree."""
import numpy as np
import pytest

from paper_2503_01840_b200 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["fp32", "bf16"])
def test_reads_after_a_plain_step_are_that_steps(dtype):
    from paper_2503_01840_b200 import binding as sb
    cfg = synth.ModelCfg("P", dtype, 2, 256, 2, 1, 128, 512, 1000, 500, (0, 1, 1), 5e5, tree_depth=3, tree_topk=4, tree_nodes=12, seed=3)
    tw, dw = synth.make_target_weights(cfg, device="cuda"), synth.make_draft_weights(cfg, device="cuda")
    prompts = [np.arange(20 + 9 * b, dtype=np.int32) * (3 + b) % cfg.vocab for b in range(3)]

    def run(batch):
        dec = sb.SpecDecoder(cfg.replace(batch=len(batch)), tw, dw, batch=len(batch), max_ctx=160, flags=sb.FLAG_CAPTURE)
        first = dec.prefill([prompts[b] for b in batch], 32)
        dec.step()                                                 # a tree's rows lie there now
        dec.prefill([prompts[b] for b in batch], 32)
        root, seen = first, []
        for _ in range(2):
            out = dec.plain_step()
            seen.append([[dec.debug(w, i) for w in (sb.DBG_TREE_TOK, sb.DBG_Y, sb.DBG_TARGET_LOGITS, sb.DBG_NODE_TAPS, sb.DBG_NODE_HIDDEN)] for i in range(len(batch))])
            for i in range(len(batch)):
                tok, y, logits = seen[-1][i][:3]
                assert tok.tolist() == [root[i]] and y.tolist() == [out[i]] and int(np.argmax(logits)) == out[i]
            root = out
        dec.close()
        return seen

    together, tol = run([0, 1, 2]), 1e-5 if dtype == "fp32" else 2e-2
    for b in range(3):
        alone = run([b])
        for i in range(2):
            for x, y in zip(together[i][b], alone[i][0]):
                assert x.shape == y.shape and np.abs(x.astype(np.float64) - y.astype(np.float64)).max() <= tol * max(1.0, np.abs(y).max()), (b, i)
