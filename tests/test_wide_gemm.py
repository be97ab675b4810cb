"""The row-major GEMM kernels of wide passes one by one, in every form, at the edges of their tiles, against the CPU oracle."""
import numpy as np
import pytest
import torch

import pyoracle as po
from paper_2503_01840_b200 import binding as sb

pytestmark = pytest.mark.gpu


def _rand(seed, *shapes):
    g = torch.Generator().manual_seed(seed)
    return [(torch.randn(*s, generator=g) / (1 if i == 0 else s[1] ** 0.5)).to(torch.bfloat16) for i, s in enumerate(shapes)]


def _same(a, b):
    return torch.equal(a.view(torch.int16 if a.dtype == torch.bfloat16 else torch.int32), b.view(torch.int16 if b.dtype == torch.bfloat16 else torch.int32))


@pytest.mark.parametrize("form", [1, 2, 3, 4])
@pytest.mark.parametrize("rows,O,I", [(1, 8, 264), (127, 136, 256), (128, 256, 320), (129, 248, 1000), (255, 512, 776), (256, 264, 4096), (257, 1024, 512),
                                      (600, 504, 1160)])
def test_row_major_gemm_vs_oracle(rows, O, I, form):
    """One to three row tiles, whole and ragged feature tiles and contractions, one to four K slices (uneven ones too)."""
    x, w = _rand(rows + O + I, (rows, I), (O, I))
    out, used = sb.gemm_wide(x.cuda(), w.cuda(), form=form)
    assert used == form
    ref = po.linear(w, x.float().numpy())
    # outputs of order 1 from exact products: fp32 sums of up to 4096 of them, in any order
    assert np.abs(out.cpu().numpy() - ref).max() < 1e-4
    assert _same(out, sb.gemm_wide(x.cuda(), w.cuda(), form=form)[0]), "the sum over the slices must be deterministic"


@pytest.mark.parametrize("form", [1, 64, 80, 128, 208, 256])
@pytest.mark.parametrize("rows,F,I", [(1, 8, 64), (128, 208, 320), (129, 1000, 264), (256, 416, 1024), (300, 520, 512), (513, 264, 136)])
def test_row_major_gate_up_vs_oracle(rows, F, I, form):
    """Tiles of 64 to 256 features per pair and the persistent kernel with 128, whole and ragged."""
    x, wg, wu = _rand(rows + F + I, (rows, I), (F, I), (F, I))
    out, used = sb.gemm_wide(x.cuda(), wg.cuda(), wu.cuda(), form=form)
    assert used == form
    xf = x.float().numpy()
    ref = po.swiglu(po.linear(wg, xf), po.linear(wu, xf))
    err = np.abs(out.float().cpu().numpy() - ref) - 2.0 ** -8 * np.abs(ref)          # one bf16 rounding of the result
    assert err.max() < 1e-4, err.max()
    assert _same(out, sb.gemm_wide(x.cuda(), wg.cuda(), wu.cuda(), form=form)[0])


@pytest.mark.parametrize("rows,O,I,up,want", [(256, 4096, 4096, False, 3), (256, 4096, 14336, False, 3), (2048, 4096, 4096, False, 1), (256, 512, 1160, False, 4),
                                              (256, 6144, 4096, False, 2), (256, 14336, 4096, True, 208), (3072, 14336, 4096, True, 1)])
def test_the_plan_takes_several_forms(rows, O, I, up, want):
    """The widths of the 8B-shaped layers run in the form with the fewest waves, and every form of the plan occurs among them."""
    x, w = (torch.zeros(n, I, dtype=torch.bfloat16, device="cuda") for n in (rows, O))
    assert sb.gemm_wide(x, w, w if up else None)[1] == want


@pytest.mark.parametrize("rows,O,I,form", [(200, 100, 256, 0), (200, 128, 252, 0), (200, 128, 64, 2), (200, 128, 256, 5), (200, 128, 512, -1)])
def test_unsupported_shapes_are_refused(rows, O, I, form):
    x, w = (torch.zeros(n, I, dtype=torch.bfloat16, device="cuda") for n in (rows, O))
    with pytest.raises(sb.SpecError):
        sb.gemm_wide(x, w, form=form)


ROWS = [8, 9, 16, 130, 152, 185, 192, 193, 208, 240]          # one row tile shared evenly by the CTAs of a pair, in whole groups of eight rows


@pytest.mark.parametrize("form", [2, 3, 4])
@pytest.mark.parametrize("rows", ROWS)
def test_one_row_tile_shared_evenly_vs_oracle(rows, form):
    x, w = _rand(rows, (rows, 1160), (264, 1160))
    out, used = sb.gemm_wide(x.cuda(), w.cuda(), form=form)
    assert used == form
    # outputs of order 1 from exact products: fp32 sums of 1160 of them, in any order
    assert np.abs(out.cpu().numpy() - po.linear(w, x.float().numpy())).max() < 1e-4


@pytest.mark.parametrize("form", [1, 64, 208])
@pytest.mark.parametrize("rows", ROWS + [300])
def test_gate_up_of_a_shared_row_tile_vs_oracle(rows, form):
    """Some rows of zeros and some whose gates leave the exponential's range among them."""
    x, wg, wu = _rand(rows + 1, (rows, 320), (424, 320), (424, 320))
    x[3], x[rows - 1] = 0.0, 300.0
    out, used = sb.gemm_wide(x.cuda(), wg.cuda(), wu.cuda(), form=form)
    assert used == form
    xf = x.float().numpy()
    with np.errstate(over="ignore"):
        g, u = po.linear(wg, xf), po.linear(wu, xf)
        ref = po.swiglu(g, u)
    # one bf16 rounding of the result, and fp32 sums of 320 products whose size the last row's values raise to 300
    mag = 1e-4 * np.maximum(1.0, np.abs(xf).max(1, keepdims=True)) * np.maximum(1.0, np.abs(u))
    assert (np.abs(out.float().cpu().numpy() - ref) - 2.0 ** -8 * np.abs(ref) - mag).max() < 0


@pytest.mark.parametrize("F,I,want", [(14336, 4096, 208), (13824, 5120, 192), (11008, 4096, 160), (28672, 8192, 208)])
def test_gate_up_widths_of_one_row_tile(F, I, want):
    """One wave (or two) of the fewest features per tile, not several waves of narrow ones; from two row tiles on the persistent kernel."""
    x, w = (torch.zeros(n, I, dtype=torch.bfloat16, device="cuda") for n in (512, F))
    assert sb.gemm_wide(x[:168].contiguous(), w, w)[1] == want
    assert sb.gemm_wide(x, w, w)[1] == 1
