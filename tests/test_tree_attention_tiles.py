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
