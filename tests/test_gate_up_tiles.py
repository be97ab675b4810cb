"""Gate/up GEMM at the feature counts whose launch takes tiles of 64 gate and 64 up features (89 to 148 tile pairs), at the
edges of its row tiles, with ragged and odd feature counts, against fp64."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("F", [11272, 11401, 14336, 18944])       # first and last count that takes them, an odd one, the 8B one
@pytest.mark.parametrize("rows,I", [(1, 200), (16, 64), (17, 1024), (60, 4096), (64, 72), (65, 320), (128, 512)])
def test_gate_up_tiles_vs_fp64(rows, I, F):
    from paper_2503_01840_b200 import binding as sb
    g = torch.Generator(device="cuda").manual_seed(rows * 31 + I + F)

    def rand(*s):
        return torch.randn(*s, generator=g, device="cuda").to(torch.bfloat16)

    x, wg, wu = rand(rows, I), rand(F, I), rand(F, I)
    wg, wu = wg * I ** -0.5, wu * I ** -0.5
    out = sb.gemm_swiglu(x, wg, wu).double()
    xd, gd, ud = x.double(), wg.double(), wu.double()
    gate, up = xd @ gd.T, xd @ ud.T
    ref = torch.nn.functional.silu(gate) * up
    # fp32 sums of I products are off by at most I 2^-24 of the sum of their magnitudes; |silu'| < 1.1, |silu(g)| <= |g|; the
    # result is rounded to bf16 (8 significant bits: off by at most half of 2^-7), expf and the division add a few 2^-23
    e = I * 2.0 ** -24
    dg, du = e * (xd.abs() @ gd.abs().T), e * (xd.abs() @ ud.abs().T)
    bound = ref.abs() * (2.0 ** -8 + 2.0 ** -18) + 1.1 * dg * (up.abs() + du) + gate.abs() * du + 1e-30
    assert bool(((out - ref).abs() <= bound).all())
