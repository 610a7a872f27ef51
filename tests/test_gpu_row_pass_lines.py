"""The row pass on blocks of 16 time steps whose chunks are whole lines, other
than the 16^3 block: chunks of 32, 160, 192 and 256 rows, more and fewer points
than the bitmap in shared memory holds."""
import numpy as np
import pytest

import oracle  # noqa: F401
from paper_2601_20113_gb300 import dls
from test_gpu_row_pass import _built, _check, _field  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu

SHAPES = [((64, 32, 16, 16), (32, 32, 16, 16)), ((96, 16, 8, 18), (96, 8, 8, 16)), ((160, 4, 4, 16), (160, 4, 4, 16)),
          ((32, 6, 5, 32), (32, 3, 1, 16)), ((48, 16, 16, 16), (16, 16, 8, 16)), ((40, 64, 8, 16), (8, 64, 8, 16))]


@pytest.mark.parametrize("dims,block", SHAPES)
@pytest.mark.parametrize("rel", [1e-2, 1e-4])
def test_shapes(dims, block, rel):
    f = _field(dims, 7)
    _check(f, dims, block, rel * float(np.ptp(f)))


@pytest.mark.parametrize("dims,block", SHAPES)
def test_nrmse(dims, block):
    _check(_field(dims, 8), dims, block, 0.5, dls.EB_NRMSE)


@pytest.mark.parametrize("dims,block", SHAPES[:3])
@pytest.mark.parametrize("spikes", [0.5, 1e5])
def test_wide_corrections(dims, block, spikes):
    _check(_field(dims, 9, spikes), dims, block, 2e-3, cap=3)
