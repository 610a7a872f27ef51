"""Float32 plans whose whole blocks are space-side, with time-side edges among
them: the field equals the oracle decoder's."""
import numpy as np
import pytest

from test_gpu_decode_paths import _built, _check, _field  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,block", [((13, 9, 5, 33), (4, 2, 1, 16)), ((12, 6, 4, 19), (2, 2, 2, 16)), ((9, 9, 3, 34), (3, 3, 1, 32))])
@pytest.mark.parametrize("codec", [0, 1])
@pytest.mark.parametrize("rel", [1e-1, 1e-3, 1e-5])
def test_space_side(dims, block, rel, codec):
    f = _field(dims, 12, 0.01)
    _check(f, dims, block, rel * float(np.ptp(f)), 8, codec)
