"""The global-basis mode where FP32 leaves a quantized value, the order of the
modes or the kept count to the FP64 definition, and at the edges of a warp's
modes and of the size scan's tiles: every record is the oracle's."""
import numpy as np
import pytest

from paper_2601_20113_gb300 import synth
from test_gpu_global import _built, _check  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


# M = 1, 8, 27, 125; two-dimensional 9, 25, 121; record counts around a tile of 1024
@pytest.mark.parametrize("dims,m", [((8, 8, 8, 2), 1), ((20, 16, 16, 2), 2), ((24, 18, 12, 7), 3), ((20, 15, 10, 6), 5),
                                    ((96, 96, 1, 1), 3), ((35, 30, 1, 9), 5), ((33, 22, 1, 5), 11), ((32, 32, 4, 16), 4)])
@pytest.mark.parametrize("eps", [3.0, 0.05])
def test_orders(dims, m, eps):
    nx, ny, nz, nt = dims
    f = synth.modes3d(nx, ny, nz, nt, seed=9, count=24).numpy()[0]
    _check(f, m, eps)


@pytest.mark.parametrize("change", ["offset", "ties", "zeros", "tiny", "huge", "outside_f32", "tight", "white"])
def test_decisions_left_to_the_definition(change):
    nx, ny, nz, nt = 16, 16, 16, 5
    f = synth.modes3d(nx, ny, nz, nt, seed=10, count=24).numpy()[0]
    eps = 1.0
    if change == "offset":
        f = f + np.float32(1000)
        eps = 1e-3
    elif change == "ties":                         # equal magnitudes
        f = np.sign(f).astype(np.float32)
        eps = 20.0
    elif change == "zeros":
        f[:, :, :8] = 0
    elif change == "tiny":
        f = (f * 1e-13).astype(np.float32)
    elif change == "huge":
        f = (f * 1e13).astype(np.float32)
    elif change == "outside_f32":                  # squares beyond FP32
        f = (f * 1e-25).astype(np.float32)
    elif change == "tight":
        eps = 1e-6
    else:                                          # every mode alike
        f = np.random.default_rng(3).standard_normal(f.shape).astype(np.float32)
        eps = 30.0
    _check(f, 4, eps)
