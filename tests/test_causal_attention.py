"""The causal tcgen05 attention kernel of training-time test against the CPU oracle, at the edges of its tiles."""
import numpy as np
import pytest
import torch

import pyoracle as po
from paper_2503_01840_b200 import binding as sb

pytestmark = pytest.mark.gpu

@pytest.mark.parametrize("T,H,G,J,ps,shift", [(1, 8, 2, 2, 16, 0), (127, 2, 2, 1, 32, 0), (256, 6, 2, 0, 64, 0), (257, 4, 4, 3, 16, 0),
                                              (385, 3, 1, 2, 16, 0), (384, 8, 2, 3, 64, 0), (200, 4, 2, 3, 16, 4), (130, 3, 3, 8, 32, 4)])
def test_causal_kernel_edges_vs_oracle(T, H, G, J, ps, shift):
    """One position, whole and ragged tiles, both ways of pairing query tiles, the three page sizes, and diagonal entries
    that start on an 8-byte boundary only (shift elements into their allocation)."""
    hd = 128
    g = torch.Generator().manual_seed(T * 7 + J)

    def rand(*s):
        return torch.randn(*s, generator=g).to(torch.bfloat16)

    q, k0, v0 = rand(T, H, hd), rand(T, G, hd), rand(T, G, hd)
    kd, vd = (rand(J, T, G, hd), rand(J, T, G, hd)) if J else (None, None)
    pages = (T + ps - 1) // ps
    perm = torch.randperm(pages + 2, generator=g)[:pages].to(torch.int32)
    kp, vp = torch.zeros(pages + 2, G, ps, hd, dtype=torch.bfloat16), torch.zeros(pages + 2, G, ps, hd, dtype=torch.bfloat16)
    for p_ in range(T):
        kp[perm[p_ // ps], :, p_ % ps] = k0[p_]
        vp[perm[p_ // ps], :, p_ % ps] = v0[p_]

    def dev(t):
        buf = torch.empty(t.numel() + shift, dtype=torch.bfloat16, device="cuda")
        buf[shift:] = t.flatten().cuda()
        return buf[shift:].view(t.shape)

    out, lse = sb.ttt_attention(q.cuda(), kp.cuda(), vp.cuda(), perm.cuda(), dev(kd) if J else None, dev(vd) if J else None, want_lse=True)
    zero = np.zeros((0, T, G, hd))
    o_out, o_lse = po.ttt_attention_rows(q.float().numpy(), k0.float().numpy(), v0.float().numpy(), kd.float().numpy() if J else zero,
                                         vd.float().numpy() if J else zero, list(range(T)))
    # outputs of order 1: bf16 output and bf16 probabilities, 2^-9 each; the statistics are fp32
    assert np.abs(out.float().cpu().numpy() - o_out).max() < 2e-2
    assert np.abs(lse.cpu().numpy() - o_lse).max() < 1e-4


@pytest.mark.parametrize("T,H,G", [(130, 4, 1), (200, 2, 2)])
def test_rows_whose_scores_are_all_minus_infinity(T, H, G):
    """An infinite query component against keys that are all negative there: the row's output is 0 and its normaliser -inf;
    the other rows are what they are without it."""
    g = torch.Generator().manual_seed(T)
    q, k, v = (torch.randn(*s, generator=g).to(torch.bfloat16).cuda() for s in ((T, H, 128), (-(-T // 16), G, 16, 128), (-(-T // 16), G, 16, 128)))
    k[..., 5] = -1.0 - k[..., 5].abs()
    table = torch.arange(k.shape[0], dtype=torch.int32, device="cuda")
    out, lse = sb.ttt_attention(q, k, v, table, None, None, want_lse=True)
    bad = torch.zeros(T, H, dtype=torch.bool, device="cuda")
    for r, h in ((0, 0), (70, 1), (T - 1, H - 1)):
        q[r, h, 5], bad[r, h] = float("inf"), True
    out2, lse2 = sb.ttt_attention(q, k, v, table, None, None, want_lse=True)
    assert (out2[bad] == 0).all() and (lse2[bad] == -float("inf")).all()
    assert torch.equal(out2[~bad], out[~bad]) and torch.equal(lse2[~bad], lse[~bad]) and torch.isfinite(lse).all()


@pytest.mark.parametrize("T,H,G,J", [(40, 2, 1, 0), (128, 4, 1, 2), (300, 2, 2, 1), (513, 4, 4, 0)])
def test_softmax_warps_that_come_late(T, H, G, J):
    """Warps that look for a tile's last contraction long after it completed (one to nine key steps per tile) find it
    complete, and the outputs are the same bits."""
    g = torch.Generator().manual_seed(T)
    pages = -(-T // 16)
    q, k, v = (torch.randn(*s, generator=g).to(torch.bfloat16).cuda() for s in ((T, H, 128), (pages, G, 16, 128), (pages, G, 16, 128)))
    kd, vd = (torch.randn(J, T, G, 128, generator=g).to(torch.bfloat16).cuda() for _ in range(2)) if J else (None, None)
    table = torch.arange(pages, dtype=torch.int32, device="cuda")
    run = lambda: sb.ttt_attention(q, k, v, table, kd, vd, want_lse=True)
    out, lse = run()
    sb.lib().spec_debug_causal(1)
    try:
        late, late_lse = run()
        torch.cuda.synchronize()
    finally:
        sb.lib().spec_debug_causal(0)
    assert torch.isfinite(lse).all() and torch.equal(out, late) and torch.equal(lse, late_lse)
