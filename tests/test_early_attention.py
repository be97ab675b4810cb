"""The attention kernels' reads ahead of the wait for the QKV launch (row metadata, page table, key tiles of nothing but context): a
step with programmatic dependent launch gives the bits that the same launches give one after the other, for contexts around the
64 keys of a tile and around the depths of the rings, and for batches in which some sequences have fewer tiles than key splits."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

CONTEXTS = (1, 62, 63, 64, 65, 127, 128, 129, 191, 193, 255, 257, 320, 321, 385, 641)


@pytest.mark.parametrize("heads,kv,hd,topk,umma", [
    (8, 2, 128, 5, 1),       # tcgen05 kernel
    (8, 2, 128, 5, 0),       # mma.sync kernel
    (8, 2, 128, 1, 2),       # few query rows: chains
    (8, 2, 64, 5, 2),
], ids=["tcgen05", "mma", "chain", "hd64"])
@pytest.mark.parametrize("batch", [1, 3])
def test_dependent_launch_equals_plain_order(heads, kv, hd, topk, umma, batch):
    from paper_2503_01840_b200 import binding as sb
    from paper_2503_01840_b200 import synth
    cfg = synth.ModelCfg("E", "bf16", 3, 512, heads, kv, hd, 1408, 2050, 1024, (0, 1, 2), 5e5, tree_depth=3, tree_topk=topk, tree_nodes=4 if topk == 1 else 24, seed=31).replace(batch=batch)
    tw, dw = synth.make_target_weights(cfg, device="cuda"), synth.make_draft_weights(cfg, device="cuda")
    decs = [sb.SpecDecoder(cfg, tw, dw, batch=batch, max_ctx=1600, flags=f, page_shuffle_seed=3) for f in (0, sb.FLAG_NO_PDL)]
    decs[0].tune(sb.SpecDecoder.TUNE_ATTN_UMMA, umma)
    try:
        for n in CONTEXTS:
            lens = [n, max(1, n // 3), 2 * n + 5][:batch]
            prompts = [np.random.default_rng(n + b).integers(0, cfg.vocab, l).astype(np.int32) for b, l in enumerate(lens)]
            seen = []
            for dec in decs:
                got = [dec.prefill(prompts, 64)]
                for _ in range(3):
                    got += dec.step() + [dec.debug(sb.DBG_NODE_HIDDEN, b) for b in range(batch)]
                got += [dec.plain_step(), *(dec.debug(sb.DBG_NODE_HIDDEN, b)[: cfg.hidden] for b in range(1))]
                seen.append(got)
            assert all(np.array_equal(x, y) for x, y in zip(*seen)), n
    finally:
        decs[0].tune(sb.SpecDecoder.TUNE_ATTN_UMMA, 2)
        for dec in decs:
            dec.close()
