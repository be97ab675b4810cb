"""The attention kernel of few query rows per KV head (chain drafts, single-token decoding): factors at the end of the fp32 range."""
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
