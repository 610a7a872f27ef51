"""The verification's sums of squares where float32's squares lose bits or
vanish, against the same sums in 64 bits."""
import pytest
import torch

from test_gpu_verify import _expect, _report

pytestmark = pytest.mark.gpu


def _check(x, y, eb):
    r = _report(x, y, eb)
    mx, over, se, sx = _expect(x, y, eb)
    assert r["max_abs_err"] == mx and r["n_over_bound"] == over
    # float pairs carry 2^-46 a point; atomics add in any order
    assert r["sum_sq_err"] == pytest.approx(se, rel=1e-12, abs=0) and r["sum_sq"] == pytest.approx(sx, rel=1e-12, abs=0)


@pytest.mark.parametrize("scale", [1e-15, 1e-19, 1e-22, 1e-25, 1e-38, 1e-44])
@pytest.mark.parametrize("shape", [(1, 1, 1, 1, 1), (2, 8, 4, 16, 20), (1, 17, 9, 33, 31), (1, 64, 16, 64, 68)])
def test_scales(scale, shape):
    gen = torch.Generator(device="cuda").manual_seed(3)
    x = (scale * torch.randn(shape, generator=gen, device="cuda", dtype=torch.float64)).float()
    y = (x.double() + 1e-3 * scale * torch.randn(shape, generator=gen, device="cuda", dtype=torch.float64)).float()
    _check(x, y, 2e-3 * scale if scale > 1e-40 else 1e-44)
    _check(x, x, scale)
    _check(x, torch.zeros_like(x), scale)


def test_small_differences_of_large_values():
    gen = torch.Generator(device="cuda").manual_seed(5)
    x = torch.randn((1, 8, 8, 32, 36), generator=gen, device="cuda")
    x[:, ::2] *= 1e-20                                # every other snapshot tiny
    y = x.clone()
    y[:, ::2] *= 1 + 2.0 ** -20
    _check(x, y, 1e-30)
    _check(torch.zeros_like(x), torch.zeros_like(x), 1e-30)
