"""Epilogues of the weight-streaming GEMM that work row by row on the summed K slices: shares of rows that do not fill a batch,
ragged feature counts, every cluster size; the top-K selection of the draft LM head; norm weights without alignment."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("split", [1, 2, 3, 5, 7, 8])
@pytest.mark.parametrize("rows,O", [(1, 130), (6, 1000), (16, 257), (17, 128), (41, 384), (60, 1001), (64, 132), (100, 256), (256, 200)])
def test_split_sums_vs_fp64(rows, O, split):
    from paper_2503_01840_b200 import binding as sb
    I = 1160                                                       # 18 k-blocks and an eighth
    g = torch.Generator(device="cuda").manual_seed(rows + O + split)
    x, w = (torch.randn(n, I, generator=g, device="cuda").to(torch.bfloat16) for n in (rows, O))
    out = sb.gemm_fused(x, w, split=split).double()
    xd, wd = x.double(), w.double()
    bound = I * 2.0 ** -24 * (xd.abs() @ wd.abs().T)               # fp32 sums of I products in any order
    assert bool(((out - xd @ wd.T).abs() <= bound).all())
    assert torch.equal(sb.gemm_fused(x, w, split=split).double(), out)


@pytest.mark.parametrize("levels", [2, 6, 40, 4000])
@pytest.mark.parametrize("rows,O,K", [(12, 130, 1), (40, 144, 15), (40, 1000, 10), (64, 32000, 3), (33, 159, 8)])
def test_topk_selection_with_ties(rows, O, K, levels):
    """Logits of few distinct values: more than 32 candidates per tile, or nearly so, or hardly any tie; a last tile of 2, 16,
    104 or 31 features.  The logits are planted exactly: x is an identity."""
    from paper_2503_01840_b200 import binding as sb
    g = torch.Generator().manual_seed(O + K + levels)
    z = (torch.randint(0, levels, (rows, O), generator=g).float() / 16 - 2).to(torch.bfloat16)
    I = (rows + 7) // 8 * 8
    x, w = torch.zeros(rows, I, dtype=torch.bfloat16), torch.zeros(O, I, dtype=torch.bfloat16)
    x[torch.arange(rows), torch.arange(rows)] = 1.0
    w[:, :rows] = z.t()
    idx, lp = sb.gemm_topk(x.cuda(), w.cuda(), K)
    order = torch.argsort(z.float(), dim=1, descending=True, stable=True)[:, :K]       # equal values: lower id first
    assert torch.equal(idx.cpu().long(), order)
    ref = torch.log_softmax(z.double(), 1).gather(1, order)
    assert float((lp.cpu().double() - ref).abs().max()) < 1e-4          # |values| up to 248: 2^-24 of them, and of sums of 32000 terms


@pytest.mark.parametrize("batch,nodes", [(1, 60), (2, 50)])
def test_norm_weights_need_no_alignment(batch, nodes):
    from paper_2503_01840_b200 import binding as sb
    from paper_2503_01840_b200 import synth
    cfg = synth.ModelCfg("N", "bf16", 2, 512, 8, 2, 128, 1408, 2050, 1024, (0, 1, 1), 5e5, tree_depth=4, tree_topk=5, seed=43).replace(batch=batch, tree_nodes=nodes)

    def shifted(t):                                                # the same values two bytes off
        buf = torch.empty(t.numel() + 1, dtype=t.dtype, device=t.device)
        buf[1:].copy_(t.view(-1))
        return buf[1:].view(t.shape)

    def off_grid(w):
        return {k: [off_grid(x) for x in v] if isinstance(v, list) else shifted(v) if "norm" in k else v for k, v in w.items()}

    tw, dw = synth.make_target_weights(cfg, device="cuda"), synth.make_draft_weights(cfg, device="cuda")
    prompts = [np.arange(9 + b, dtype=np.int32) * 7 % cfg.vocab for b in range(batch)]
    seen = []
    for t, d in ((tw, dw), (off_grid(tw), off_grid(dw))):
        dec = sb.SpecDecoder(cfg, t, d, batch=batch, max_ctx=128)
        got = [dec.prefill(prompts, 16)]
        got += [x for _ in range(2) for x in dec.step()]
        got += [dec.debug(sb.DBG_NODE_HIDDEN, b) for b in range(batch)]
        seen.append(got)
        dec.close()
    assert all(np.array_equal(x, y) for x, y in zip(*seen)) and np.isfinite(seen[0][-1]).all()
