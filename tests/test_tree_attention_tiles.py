"""The tcgen05 tree attention kernel at every number of key tiles per CTA around its rings (score buffers, stages), ragged ends
and one or two query tiles, against fp64."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows", [5, 40])                    # 20 and 160 query rows per KV head
@pytest.mark.parametrize("ctx", [0, 40, 64, 100, 190, 256, 300, 385, 505, 640, 770, 830, 1100, 1407])
def test_tree_attention_tiles_vs_fp64(rows, ctx):
    from paper_2503_01840_b200 import binding as sb
    H, G, hd, ps, tail = 8, 2, 128, 16, rows
    n = ctx + tail
    pages = (n + ps - 1) // ps
    g = torch.Generator(device="cuda").manual_seed(ctx + rows)

    def rand(*s):
        return torch.randn(*s, generator=g, device="cuda").to(torch.bfloat16)

    q, kp, vp = rand(rows, H, hd) * 2, rand(pages, G, ps, hd), rand(pages, G, ps, hd)
    table = torch.randperm(pages, generator=g, device="cuda").to(torch.int32).view(1, -1)
    vis = torch.rand(rows, tail, generator=g, device="cuda") < 0.5
    vis[:, 0] = True
    lo = torch.tensor([sum(1 << t for t in range(tail) if vis[r, t]) for r in range(rows)], dtype=torch.int64, device="cuda")
    full = lambda c: torch.full((rows,), c, dtype=torch.int32, device="cuda")
    # a hint of one tile beside the tail's: two key splits whatever the context is
    out = sb.attention(q, kp, vp, table, ps, full(0), full(ctx), full(ctx), lo, torch.zeros_like(lo), tail, G, 64, impl=3).double()
    K, V = (p[table[0].long()].permute(1, 0, 2, 3).reshape(G, pages * ps, hd)[:, :n].double() for p in (kp, vp))
    s = torch.einsum("rgch,gnh->rgcn", q.double().view(rows, G, H // G, hd), K) * hd ** -0.5
    mask = torch.cat([torch.ones(rows, ctx, dtype=torch.bool, device="cuda"), vis], 1)
    p = s.masked_fill(~mask[:, None, None], -np.inf).softmax(-1)
    ref = torch.einsum("rgcn,gnh->rgch", p, V).reshape(rows, H, hd)
    mag = torch.einsum("rgcn,gnh->rgch", p, V.abs()).reshape(rows, H, hd)
    # the probabilities and the result are rounded to bf16 (8 significant bits), everything else is fp32
    assert bool(((out - ref).abs() <= 2.0 ** -8 * 1.01 * (mag + ref.abs()) + 1e-5).all())


@pytest.mark.parametrize("rows,grp,ctx", [(1, 20, 100), (5, 4, 700), (33, 4, 64), (37, 5, 300), (64, 8, 1500)])
def test_rows_out_alignment_and_padding_queries(rows, grp, ctx):
    """tcgen05 kernel, rows per tile that fill it, leave warps without rows or need several tiles, one and several key splits: against
    fp64; padding rows (whatever their queries hold) give zeros; the same bits where out and scratch take no vector stores."""
    from paper_2503_01840_b200 import binding as sb
    G, hd, ps, tail = 2, 128, 16, 3
    H, pps = G * grp, (ctx + tail + 15) // 16
    g = torch.Generator(device="cuda").manual_seed(rows + ctx)
    q, kp, vp = (torch.randn(*s, generator=g, device="cuda").to(torch.bfloat16) for s in ((rows, H, hd), (pps, G, ps, hd), (pps, G, ps, hd)))
    seq = torch.zeros(rows, device="cuda", dtype=torch.int32)
    if rows > 4:
        seq[2] = seq[rows - 1] = -1
        q[2], q[rows - 1] = float("nan"), float("inf")
    table = torch.randperm(pps, generator=g, device="cuda").to(torch.int32).view(1, pps)
    c = torch.full((rows,), ctx, device="cuda", dtype=torch.int32)
    lo = torch.randint(0, 8, (rows,), generator=g, device="cuda") | 1
    hi = torch.zeros_like(lo)
    need = sb.lib().spec_attn_scratch_bytes(rows, H, hd, ctx)
    got = []
    for off in (0, 1, 4):
        out = torch.full((rows * H * hd + 8,), 5.0, device="cuda", dtype=torch.bfloat16)
        scratch = torch.empty(need + 16, device="cuda", dtype=torch.uint8)
        assert sb.lib().spec_attention(1, 3, q.data_ptr(), kp.data_ptr(), vp.data_ptr(), table.data_ptr(), pps, ps, seq.data_ptr(), c.data_ptr(), c.data_ptr(),
                                       lo.data_ptr(), hi.data_ptr(), tail, out.data_ptr() + 2 * off, rows, H, G, hd, ctx, scratch.data_ptr() + 8 * (off > 0),
                                       torch.cuda.current_stream().cuda_stream) == 0
        torch.cuda.synchronize()
        assert bool((out[:off] == 5.0).all()) and bool((out[off + rows * H * hd:] == 5.0).all())
        got.append(out[off:off + rows * H * hd])
    assert all(torch.equal(got[0], o) for o in got[1:])
    K, V = (p[table[0].long()].permute(1, 0, 2, 3).reshape(G, pps * ps, hd)[:, : ctx + tail].double() for p in (kp, vp))
    o = got[0].view(rows, H, hd).double()
    for r in range(rows):
        if int(seq[r]) < 0:
            assert not o[r].any()
            continue
        seen = list(range(ctx)) + [ctx + t for t in range(tail) if int(lo[r]) >> t & 1]
        p = (torch.einsum("gch,gnh->gcn", q[r].double().view(G, grp, hd), K[:, seen]) * hd ** -0.5).softmax(-1)
        ref, mag = (torch.einsum("gcn,gnh->gch", p, x[:, seen]).reshape(H, hd) for x in (V, V.abs()))
        # probabilities up to 2^8 times the sum's unit and the result are rounded to bf16 (8 significant bits), the rest is fp32
        assert bool(((o[r] - ref).abs() <= 2.0 ** -8 * 1.01 * (mag + ref.abs()) + 1e-5).all()), r
