"""The verification's sums of squares at the ends of float32's range, against
the same sums in 64 bits."""
import math

import pytest
import torch

from test_gpu_verify import _report

pytestmark = pytest.mark.gpu

SHAPES = [(1, 1, 1, 1, 1), (1, 1, 1, 16, 16), (1, 1, 1, 16, 17), (1, 8, 16, 64, 68)]


# one difference of 2^60 + 2^36 everywhere (a float and its rounding error, the
# latter's square past the pairs): the 64-bit sums of up to 256 points, one a
# thread, are exact
@pytest.mark.parametrize("shape", SHAPES)
def test_large_differences(shape):
    n = math.prod(shape)
    x = torch.full(shape, 2.0 ** 60, device="cuda")
    y = torch.full(shape, -(2.0 ** 36), device="cuda")
    d = 2.0 ** 60 + 2.0 ** 36
    r = _report(x, y, 1.0)
    assert r["max_abs_err"] == d and r["n_over_bound"] == n
    # beyond them a rounding of 2^-53 an addition: up to 1 024 of a thread, 5 of a warp, 9 728 warps
    rel = 2.0 ** -51 if n <= 256 else 1.5e-12
    assert r["sum_sq_err"] == pytest.approx(n * d * d, rel=rel, abs=0)
    assert r["sum_sq"] == pytest.approx(n * 2.0 ** 120, rel=rel, abs=0)
