"""The verification report over alignments, sizes around its loads and
batches, values beyond FP32's squares and points on the bound, against the
same quantities in 64 bits."""
import math

import numpy as np
import pytest
import torch

from paper_2601_20113_gb300 import dls

pytestmark = pytest.mark.gpu


def _report(x, y, eb, eb_type=dls.EB_ABS):
    """Of fields x and y (nvars, nt, nz, ny, nx) against a stream that carries the bound eb."""
    comp = dls.compress(torch.zeros_like(x), (1, 1, 1, 1), eb, eb_type)
    return dls.verify(x, y, comp)


def _expect(x, y, eb):
    x, y = x.cpu().double(), y.cpu().double()
    d = (x - y).abs()
    return d.max().item(), int((d > eb).sum()), math.fsum((d.numpy().ravel() ** 2).tolist()), math.fsum((x.numpy().ravel() ** 2).tolist())


def _check(x, y, eb):
    r = _report(x, y, eb)
    mx, over, se, sx = _expect(x, y, eb)
    assert r["max_abs_err"] == mx and r["n_over_bound"] == over and r["status"] == (-7 if over else 0)
    # float pairs carry 2^-46 a point; atomics add in any order
    assert r["sum_sq_err"] == pytest.approx(se, rel=1e-12) and r["sum_sq"] == pytest.approx(sx, rel=1e-12)


@pytest.mark.parametrize("shape", [(1, 1, 1, 1, 1), (1, 1, 1, 3, 5), (2, 3, 1, 7, 9), (1, 17, 9, 33, 31), (1, 16, 16, 64, 68)])
@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("offset", [0, 1])
def test_sizes_and_alignment(shape, dtype, offset):
    n = int(np.prod(shape))
    gen = torch.Generator(device="cuda").manual_seed(n)
    b = torch.randn(2 * n + 2, generator=gen, device="cuda", dtype=torch.float64).to(dtype)
    x = b[offset:offset + n].view(shape)
    y = (x + 1e-3 * torch.randn(shape, generator=gen, device="cuda", dtype=torch.float64).to(dtype))
    _check(x, y, 2e-3)


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("scale", [1e-12, 1.0, 1e19, 1e30])
def test_scales_and_points_on_the_bound(dtype, scale):
    if dtype == torch.float64 and scale == 1e30:
        scale = 1e150
    gen = torch.Generator(device="cuda").manual_seed(3)
    x = (scale * torch.randn((1, 8, 4, 16, 20), generator=gen, device="cuda", dtype=torch.float64)).to(dtype)
    eb = float(torch.tensor(scale * 1e-2, dtype=dtype))
    y = x.clone()
    f = y.view(-1)
    f[::7] += eb                         # on the bound up to the addition's rounding
    f[::11] -= 3 * eb
    _check(x, y, eb)
    _check(x, x, eb)                     # nothing differs
    _check(x, torch.zeros_like(x), eb)   # nearly every point is over


def test_non_finite_points():
    x = torch.ones((1, 4, 4, 8, 8), device="cuda")
    y = x.clone()
    y.view(-1)[5] = float("nan")
    y.view(-1)[9] = 1.5
    r = _report(x, y, 0.25)
    assert r["max_abs_err"] == 0.5 and r["n_over_bound"] == 1 and math.isnan(r["sum_sq_err"]) and r["sum_sq"] == 1024
    y.view(-1)[5] = float("inf")
    r = _report(x, y, 0.25)
    assert r["max_abs_err"] == float("inf") and r["n_over_bound"] == 2
