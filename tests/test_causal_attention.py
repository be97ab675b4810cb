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
