"""The fp32 model's GEMM and attention kernels at the edges of their row groups, against fp64."""
import numpy as np
import pytest
import torch

from paper_2503_01840_b200 import binding as sb

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows,O,I,shift", [(1, 1, 4, 0), (3, 31, 128, 0), (4, 256, 256, 0), (5, 33, 688, 0), (8, 8, 12, 0), (9, 1000, 260, 0),
                                            (16, 100, 768, 0), (17, 65, 132, 0), (32, 7, 512, 0), (33, 300, 256, 0), (256, 64, 128, 0),
                                            (257, 64, 128, 0), (64, 2049, 2052, 0), (4, 50, 30, 0), (4, 50, 32, 1),
                                            (256, 4096, 64, 0), (17, 16390, 32, 0), (16, 33000, 16, 0)])
def test_fp32_gemm_row_groups(rows, O, I, shift):
    """Every row group of the warp-per-feature kernel, its remainders, and the shapes that stay on the tile kernel (a
    contraction that is no multiple of four, operands off a 16-byte boundary, many rows of a large weight, a contraction that is
    short for its many outputs)."""
    g = torch.Generator().manual_seed(rows * 1000 + O + I)
    x, w = torch.randn(rows, I, generator=g), torch.randn(O, I, generator=g)

    def dev(t):
        buf = torch.empty(t.numel() + shift, device="cuda")
        buf[shift:] = t.flatten().cuda()
        return buf[shift:].view(t.shape)

    out = sb.gemm(dev(x), dev(w), impl=1).cpu().double().numpy()
    ref = x.double().numpy() @ w.double().numpy().T
    bound = 2.0 ** -23 * (8 + I / 32) * (np.abs(x.double().numpy()) @ np.abs(w.double().numpy()).T)     # 32 partial sums of I / 32 products
    assert (np.abs(out - ref) <= bound + 1e-30).all(), np.abs(out - ref).max()


@pytest.mark.parametrize("H,G,hd,ctx,tail,ps", [(4, 2, 64, 0, 1, 16), (4, 2, 64, 70, 5, 16), (2, 2, 16, 31, 33, 8), (3, 1, 128, 129, 70, 32), (2, 1, 240, 40, 128, 16)])
def test_fp32_attention_vs_fp64(H, G, hd, ctx, tail, ps):
    rows = 5
    g = torch.Generator().manual_seed(hd + ctx)
    n = ctx + tail
    pages = (n + ps - 1) // ps
    q, k, v = torch.randn(rows, H, hd, generator=g), torch.randn(n, G, hd, generator=g), torch.randn(n, G, hd, generator=g)
    perm = torch.randperm(pages + 1, generator=g)[:pages].to(torch.int32)
    kp, vp = torch.zeros(pages + 1, G, ps, hd), torch.zeros(pages + 1, G, ps, hd)
    for p in range(n):
        kp[perm[p // ps], :, p % ps], vp[perm[p // ps], :, p % ps] = k[p], v[p]
    bits = [int(b) for b in torch.randint(0, 2, (rows, 128), generator=g).flatten()]
    mask = np.array(bits, bool).reshape(rows, 128)
    mask[:, 0] = True
    words = [[int(sum(1 << i for i in range(64) if mask[r, 64 * w + i])) for r in range(rows)] for w in (0, 1)]
    lo, hi = (torch.tensor(np.array(w, np.uint64).view(np.int64)).cuda() for w in words)
    full = lambda c: torch.full((rows,), c, dtype=torch.int32, device="cuda")
    out = sb.attention(q.cuda(), kp.cuda(), vp.cuda(), perm.view(1, -1).cuda(), ps, full(0), full(ctx), full(ctx), lo, hi, tail, G, ctx + tail, impl=1)
    vis = np.concatenate([np.ones((rows, ctx), bool), mask[:, :tail]], 1)
    qd, kd, vd = q.double().numpy(), k.double().numpy(), v.double().numpy()
    for h in range(H):
        s = qd[:, h] @ kd[:, h // (H // G)].T / np.sqrt(hd)
        s[~vis] = -np.inf
        p = np.exp(s - s.max(1, keepdims=True))
        ref = (p / p.sum(1, keepdims=True)) @ vd[:, h // (H // G)]
        assert np.abs(out[:, h].cpu().double().numpy() - ref).max() < 5e-6          # scores of order 1 .. 3 in fp32, sums of ~200 terms


@pytest.mark.parametrize("dtype,tol", [(torch.float32, 5e-6), (torch.bfloat16, 2e-2)])
@pytest.mark.parametrize("hd", [512, 528, 576, 1040])
def test_plain_attention_wide_heads_vs_fp64(hd, dtype, tol):
    """Head dimensions around and above four times the threads of a CTA, where a thread owns several groups of dimensions."""
    rows, H, G, ctx, tail, ps = 3, 2, 1, 37, 3, 16
    g = torch.Generator().manual_seed(hd)
    pages = (ctx + tail + ps - 1) // ps
    q, kp, vp = (torch.randn(*s, generator=g).to(dtype) for s in ((rows, H, hd), (pages, G, ps, hd), (pages, G, ps, hd)))
    full = lambda c: torch.full((rows,), c, dtype=torch.int32, device="cuda")
    lo, hi = torch.full((rows,), 7, dtype=torch.int64, device="cuda"), torch.zeros(rows, dtype=torch.int64, device="cuda")
    table = torch.arange(pages, dtype=torch.int32, device="cuda").view(1, -1)
    out = sb.attention(q.cuda(), kp.cuda(), vp.cuda(), table, ps, full(0), full(ctx), full(ctx), lo, hi, tail, G, ctx + tail, impl=1)
    k, v = (t.double()[:, 0].reshape(pages * ps, hd)[: ctx + tail] for t in (kp, vp))
    ref = torch.softmax(q.double() @ k.T / hd ** 0.5, -1) @ v
    # fp32: scores of order 1 .. 3 and sums of 40 terms; bf16: one rounding of outputs of order 1
    assert (out.cpu().double() - ref).abs().max() < tol


@pytest.mark.parametrize("hd,ps", [(64, 16), (48, 5)])
@pytest.mark.parametrize("n", [1, 63, 64, 127, 128, 129, 255, 256, 257, 600])
def test_plain_attention_key_counts_vs_fp64(n, hd, ps):
    """Around the keys whose values are requested ahead of their scores, a round of keys, and page sizes that are no power of two."""
    H, G = 3, 1
    g = torch.Generator().manual_seed(n)
    pages = (n + ps - 1) // ps
    q, kp, vp = (torch.randn(*s, generator=g) for s in ((2, H, hd), (pages, G, ps, hd), (pages, G, ps, hd)))
    full = lambda c: torch.full((2,), c, dtype=torch.int32, device="cuda")
    lo, hi = torch.ones(2, dtype=torch.int64, device="cuda"), torch.zeros(2, dtype=torch.int64, device="cuda")
    table = torch.randperm(pages, generator=g).to(torch.int32).view(1, pages)
    out = sb.attention(q.cuda(), kp.cuda(), vp.cuda(), table.cuda(), ps, full(0), full(n - 1), full(n - 1), lo, hi, 1, G, n, impl=1).cpu().double()
    k, v = (t[table[0].long()].double()[:, 0].reshape(pages * ps, hd)[:n] for t in (kp, vp))
    ref = torch.softmax(q.double() @ k.T / hd ** 0.5, -1) @ v
    assert (out - ref).abs().max() < 5e-6                   # scores of order 1 .. 3 in fp32, sums of up to 600 terms


@pytest.mark.parametrize("K", [1, 4, 16])
@pytest.mark.parametrize("n", [16, 17, 255, 257, 1023, 1024, 1025, 2047, 2048, 2049])
def test_log_softmax_top_k_edges(n, K):
    """Numbers of logits around what a thread keeps in registers, with ties, infinities and rows of equal values."""
    g = torch.Generator().manual_seed(n + K)
    z = torch.randn(6, n, generator=g)
    z[1] = 0.25
    z[2, n // 2:] = float("-inf")
    z[3] = torch.randint(0, 3, (n,), generator=g).float()
    idx, lp = (t.cpu() for t in sb.logsoftmax_topk(z.cuda(), K, two_stage=False))
    for r in range(6):
        want = sorted(range(n), key=lambda i: (-float(z[r, i]), i))[:K]
        ref = torch.log_softmax(z[r].double(), 0)[want]
        live = [c for c in range(K) if z[r, want[c]] > float("-inf")]
        gaps = torch.diff(z[r][want]).abs()
        if not bool(((gaps > 0) & (gaps < 1e-5)).any()):    # values that fp32 log-probabilities may merge
            assert idx[r].tolist() == want, r
        assert (lp[r][live] - ref[live]).abs().max() < 1e-5


@pytest.mark.parametrize("hd,ps,dtype,tol,off", [(64, 16, torch.float32, 5e-6, 0), (48, 5, torch.float32, 5e-6, 1), (80, 16, torch.bfloat16, 2e-2, 0), (32, 16, torch.bfloat16, 2e-2, 1),
                                                 (528, 16, torch.float32, 5e-6, 0)])
@pytest.mark.parametrize("n", [1, 31, 33, 129, 600])
@pytest.mark.parametrize("rows", [197, 198])
def test_plain_attention_of_more_than_two_waves_vs_fp64(rows, n, hd, ps, dtype, tol, off):
    """591 and 594 CTAs: the last grid that reads values ahead of their scores and the first that does not.  Rows of three sequences,
    some of them padding, masks that hide tail keys (whose values hold anything); caches off their vector alignment."""
    H, G, tail = 3, 1, min(n, 4)
    ctx = n - tail
    g = torch.Generator().manual_seed(n)
    pages = (n + ps - 1) // ps
    q, kp, vp = (torch.randn(*s, generator=g).to(dtype) for s in ((rows, H, hd), (3 * pages, G, ps, hd), (3 * pages, G, ps, hd)))
    table = torch.randperm(3 * pages, generator=g).to(torch.int32).view(3, pages)
    if n > 1:                                                       # the third tail key of the last sequence is hidden from all its rows
        vp[int(table[2, (ctx + 2) // ps]), :, (ctx + 2) % ps] = float("nan")
    seq = (torch.arange(rows) % 4 - 1).to(torch.int32)              # -1: padding
    full = torch.full((rows,), ctx, dtype=torch.int32)
    lo = torch.full((rows,), 0b1011 if n > 1 else 1, dtype=torch.int64)
    kd, vd = (torch.cat([torch.zeros(off, dtype=dtype), t.flatten()]).cuda()[off:].view(t.shape) for t in (kp, vp))
    out = sb.attention(q.cuda(), kd, vd, table.cuda(), ps, seq.cuda(), full.cuda(), full.cuda(), lo.cuda(), torch.zeros_like(lo).cuda(), tail, G, n,
                       impl=1).cpu().double()
    assert not out[seq < 0].any()
    seen = [j for j in range(n) if j < ctx or 0b1011 >> (j - ctx) & 1]
    for s in range(3):
        k, v = (t[table[s].long()].double()[:, 0].reshape(pages * ps, hd)[seen] for t in (kp, vp))
        ref = torch.softmax(q[seq == s].double() @ k.T / hd ** 0.5, -1) @ v
        assert (out[seq == s] - ref).abs().max() < tol              # scores of order 1 .. 3 in fp32, sums of up to 600 terms; bf16: the output's rounding


@pytest.mark.parametrize("rows,short", [(1, 12), (1, 0), (600, 12), (600, 0)])
def test_plain_attention_takes_as_many_keys_as_shared_memory_holds(rows, short):
    """227 KB are a score per key, a query and 16 bytes: no form refuses what another takes.  (The keys a launch allows for, not those it has.)"""
    hd, ps = 64, 16
    most = (227 * 1024 - 16) // 4 - hd - 1 - short
    g = torch.Generator().manual_seed(1)
    q, kp, vp = (torch.randn(*s, generator=g) for s in ((rows, 1, hd), (2, 1, ps, hd), (2, 1, ps, hd)))
    full = torch.full((rows,), 20, dtype=torch.int32, device="cuda")
    lo = torch.ones(rows, dtype=torch.int64, device="cuda")
    out = sb.attention(q.cuda(), kp.cuda(), vp.cuda(), torch.tensor([[1, 0]], dtype=torch.int32, device="cuda"), ps, torch.zeros_like(full), full, full, lo,
                       torch.zeros_like(lo), 1, 1, most, impl=1).cpu().double()
    k, v = (t.flip(0).double().reshape(2 * ps, hd)[:21] for t in (kp, vp))
    assert (out[:, 0] - torch.softmax(q[:, 0].double() @ k.T / hd ** 0.5, -1) @ v).abs().max() < 5e-6
