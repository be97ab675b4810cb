"""The attention kernel of few query rows per KV head (chain drafts, single-token decoding) against fp64: numbers of sequences that
leave the chip idle or fill it several times, ragged contexts, factors at the end of the fp32 range."""
import math

import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("new_key", [4.0, 16.0, 32.0, 34.0])       # 16, 65, 131 and 139 powers of two between the two maxima
def test_rescaling_by_small_factors(new_key):
    """A key of score 0 with a value of 2^126 comes first, a key of a far larger score with the value 0 one tile later: the factor
    the first tile's sum is rescaled by lies below the normal fp32 range in the last two cases, its product with the sum does not."""
    from paper_2503_01840_b200 import binding as sb
    n, G, hd, ps, ctx = 40, 4, 128, 16, 127                        # 160 CTAs: both key tiles of a sequence in one of them
    pages = 8
    k, v = torch.zeros(pages, G, ps, hd), torch.zeros(pages, G, ps, hd)
    v[0, :, 0] = 2.0 ** 126
    k[4, :, 0, 0] = new_key                                        # position 64
    q = torch.zeros(n, G, hd)
    q[..., 0] = 32.0
    bf = lambda t: t.to(torch.bfloat16).cuda()
    full = lambda c: torch.full((n,), c, dtype=torch.int32, device="cuda")
    lo = torch.ones(n, dtype=torch.int64, device="cuda")
    table = torch.arange(pages, dtype=torch.int32, device="cuda").repeat(n, 1)
    out = sb.attention(bf(q), bf(k), bf(v), table, ps, torch.arange(n, dtype=torch.int32, device="cuda"), full(ctx), full(ctx), lo,
                       torch.zeros_like(lo), 1, G, ctx, impl=2).double()
    s = 32.0 * new_key / math.sqrt(hd)
    ref = 2.0 ** 126 * math.exp(-s) / (1.0 + 127 * math.exp(-s))
    # the result is rounded to bf16: 8 significant bits, half a unit is up to 2^-8 of the value; the smallest factor, 2^-138.7, has
    # 11 bits, and its exponent is off by some 2^-15
    assert float((out - ref).abs().max()) <= (2.0 ** -8 + 2.0 ** -11 + 2.0 ** -14) * ref


@pytest.mark.parametrize("hd,grp", [(128, 1), (128, 4), (128, 16), (64, 4)])
@pytest.mark.parametrize("n", [1, 5, 20, 70])
def test_ragged_sequences_vs_fp64(n, hd, grp):
    from paper_2503_01840_b200 import binding as sb
    G, ps, tail = 8, 16, 3
    H = G * grp
    g = torch.Generator(device="cuda").manual_seed(n * grp + hd)

    def rand(*s):
        return torch.randn(*s, generator=g, device="cuda").to(torch.bfloat16)

    ctx = torch.randint(0, 400, (n,), generator=g, device="cuda", dtype=torch.int32)
    ctx[0] = 399
    pps = 26
    q, kp, vp = rand(n, H, hd) * 2, rand(n * pps, G, ps, hd), rand(n * pps, G, ps, hd)
    table = torch.randperm(n * pps, generator=g, device="cuda").to(torch.int32).view(n, pps)
    lo = torch.randint(0, 8, (n,), generator=g, device="cuda") | 1                    # tail keys in sight
    out = sb.attention(q, kp, vp, table, ps, torch.arange(n, dtype=torch.int32, device="cuda"), ctx, ctx, lo, torch.zeros_like(lo), tail, G,
                       400, impl=2).double()
    for b in range(n):
        c = int(ctx[b])
        seen = torch.tensor(list(range(c)) + [c + t for t in range(tail) if int(lo[b]) >> t & 1], device="cuda")
        K, V = (p[table[b].long()].permute(1, 0, 2, 3).reshape(G, pps * ps, hd)[:, seen].double() for p in (kp, vp))
        p = (torch.einsum("gch,gnh->gcn", q[b].double().view(G, grp, hd), K) * hd ** -0.5).softmax(-1)
        ref, mag = (torch.einsum("gcn,gnh->gch", p, x).reshape(H, hd) for x in (V, V.abs()))
        # the probabilities and the result are rounded to bf16 (8 significant bits), everything else is fp32
        assert bool(((out[b] - ref).abs() <= 2.0 ** -8 * 1.01 * (mag + ref.abs()) + 1e-5).all()), b


@pytest.mark.parametrize("hd,grp,n", [(128, 4, 1), (128, 5, 3), (128, 16, 40), (64, 4, 2)])
def test_output_and_scratch_off_the_vector_alignment(hd, grp, n):
    """Results and partial results leave in vector stores where the caller's pointers allow it, else value by value: the same bits.
    (The scratch owes its statistics 8 bytes.)  Splits of one tile and of several, one split, 4 to 16 query rows."""
    from paper_2503_01840_b200 import binding as sb
    G, ps, ctx, pps = 2, 16, 700, 46
    H = G * grp
    g = torch.Generator(device="cuda").manual_seed(7)
    q, kp, vp = (torch.randn(*s, generator=g, device="cuda").to(torch.bfloat16) for s in ((n, H, hd), (n * pps, G, ps, hd), (n * pps, G, ps, hd)))
    table = torch.arange(n * pps, device="cuda", dtype=torch.int32).view(n, pps)
    seq = torch.arange(n, device="cuda", dtype=torch.int32)
    c = torch.full((n,), ctx, device="cuda", dtype=torch.int32)
    lo, hi = torch.ones(n, device="cuda", dtype=torch.int64), torch.zeros(n, device="cuda", dtype=torch.int64)
    need = sb.lib().spec_attn_scratch_bytes(n, H, hd, ctx)
    got = []
    for out_off, scratch_off in ((0, 0), (1, 0), (2, 8), (4, 8)):
        out = torch.zeros(n * H * hd + 8, device="cuda", dtype=torch.bfloat16)
        scratch = torch.empty(need + 16, device="cuda", dtype=torch.uint8)
        rc = sb.lib().spec_attention(1, 2, q.data_ptr(), kp.data_ptr(), vp.data_ptr(), table.data_ptr(), pps, ps, seq.data_ptr(), c.data_ptr(), c.data_ptr(),
                                     lo.data_ptr(), hi.data_ptr(), 1, out.data_ptr() + 2 * out_off, n, H, G, hd, ctx, scratch.data_ptr() + scratch_off,
                                     torch.cuda.current_stream().cuda_stream)
        assert rc == 0
        torch.cuda.synchronize()
        assert not out[:out_off].any() and not out[out_off + n * H * hd:].any()
        got.append(out[out_off:out_off + n * H * hd])
    assert all(torch.equal(got[0], o) for o in got[1:])


@pytest.mark.parametrize("tiles", [2, 6, 7, 18, 19, 32, 40])
@pytest.mark.parametrize("hd", [64, 128])
def test_merge_of_many_splits(hd, tiles):
    """One KV head: as many key splits as tiles, up to 32.  Around the numbers the merge takes in one go (6 and 18)."""
    from paper_2503_01840_b200 import binding as sb
    H, G, ps, ctx = 5, 1, 16, 64 * tiles - 1
    pps = 4 * tiles + 1
    g = torch.Generator(device="cuda").manual_seed(tiles)
    q, kp, vp = (torch.randn(*s, generator=g, device="cuda").to(torch.bfloat16) for s in ((1, H, hd), (pps, G, ps, hd), (pps, G, ps, hd)))
    table = torch.randperm(pps, generator=g, device="cuda").to(torch.int32).view(1, pps)
    c, lo = torch.full((1,), ctx, device="cuda", dtype=torch.int32), torch.ones(1, device="cuda", dtype=torch.int64)
    out = sb.attention(q, kp, vp, table, ps, torch.zeros(1, device="cuda", dtype=torch.int32), c, c, lo, torch.zeros_like(lo), 1, G, ctx, impl=2).double()
    K, V = (p[table[0].long()].reshape(pps * ps, hd)[: ctx + 1].double() for p in (kp, vp))
    p = (q[0].double() @ K.T * hd ** -0.5).softmax(-1)
    ref, mag = p @ V, p @ V.abs()
    assert bool(((out[0] - ref).abs() <= 2.0 ** -8 * 1.01 * (mag + ref.abs()) + 1e-5).all())       # as above
