"""The plain form where its FP32 and reciprocal tests leave a decision to the
FP64 definition, and at the edges of its row and column splits: streams stay
byte-identical to the oracle's."""
import numpy as np
import pytest
import torch

import oracle
from paper_2601_20113_gb300 import dls

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    oracle.build()


def _smooth(dims, seed, dtype):
    nx, ny, nz, nt = dims
    r = np.random.default_rng(seed)
    t, z, y, x = np.meshgrid(*[np.arange(n) / 16.0 for n in (nt, nz, ny, nx)], indexing="ij")
    f = np.zeros((nt, nz, ny, nx))
    for _ in range(5):
        k = r.uniform(0.2, 2.0, 4)
        f += r.uniform(0.2, 1.0) * np.sin(k[0] * t + k[1] * z + k[2] * y + k[3] * x + r.uniform(0, 6.28))
    f += 1e-3 * r.standard_normal(f.shape)
    return f[None].astype(dtype)


def _check(f, dims, block, eb, eb_type=oracle.EB_ABS, rank_cap=16):
    d = oracle.F32 if f.dtype == np.float32 else oracle.F64
    st, ref, _ = oracle.compress(oracle.Config(dims, block, d, eb=eb, eb_type=eb_type, rank_cap=rank_cap), f)
    assert st == 0
    got = dls.compress(torch.from_numpy(f).cuda(), block=block, eb=eb, eb_type=eb_type, rank_cap=rank_cap).cpu().numpy()
    assert got.size == ref.size and np.array_equal(got, ref)


# rows below, at and past the CTA's 256 threads and off its chunks of 32; odd orders; space-side blocks; order 32
BLOCKS = [((24, 20, 6, 18), (8, 8, 3, 16)), ((32, 32, 2, 20), (16, 16, 1, 7)), ((21, 13, 5, 13), (7, 6, 5, 13)),
          ((12, 10, 4, 64), (3, 3, 1, 40)), ((40, 20, 1, 32), (9, 7, 1, 32)), ((40, 24, 3, 33), (20, 13, 1, 31)),
          ((10, 9, 3, 9), (5, 3, 1, 1)), ((34, 34, 1, 17), (17, 17, 1, 17))]


@pytest.mark.parametrize("dims,block", BLOCKS)
@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("rel", [1e-2, 1e-4])
def test_block_edges(dims, block, dtype, rel):
    f = _smooth(dims, 3, dtype)
    _check(f, dims, block, rel * float(f.max() - f.min()), rank_cap=32)


DIMS, BLOCK = (32, 16, 17, 32), (16, 16, 16, 16)


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("change", ["offset", "tight", "zeros", "tiny", "huge", "halves", "spike"])
def test_decisions_left_to_the_definition(dtype, change):
    f = _smooth(DIMS, 4, dtype)
    eb = 1e-3 * float(f.max() - f.min())
    if change == "offset":                     # coefficients large against delta
        f = (f + 5000).astype(dtype)
    elif change == "tight":                    # near the type's own resolution: overflow, escapes, raw blocks
        eb *= 1e-5
    elif change == "zeros":
        f[:, :, 3:9] = 0
        f[:, :16, :, :, :16] = 0
    elif change == "tiny":
        f, eb = (f * 1e-33).astype(dtype), eb * 1e-33
    elif change == "huge":
        f, eb = (f * 1e25).astype(dtype), eb * 1e25
    elif change == "halves":                   # residuals and coefficients on the quantizer's ties
        f = (np.round(f * 8) / 8).astype(dtype)
        eb = 0.125
    else:
        f[0, 5, 2, 3, 4] = 1e4
    _check(f, DIMS, BLOCK, eb)


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
def test_bound_at_the_error_itself(dtype):
    """eps_l^2 placed on an exact E(r): the estimate cannot decide."""
    r = np.random.default_rng(9)
    f = (r.integers(-3, 4, (1, 16, 16, 16, 16))).astype(dtype)      # white: E(0) = sum of squares, exact
    eb = float(np.sqrt(np.square(f.astype(np.float64)).sum() / f.size))
    for e in (eb, np.nextafter(eb, 0), np.nextafter(eb, 9)):
        _check(f, (16, 16, 16, 16), BLOCK, float(e))
