"""Float32 blocks of more points than the persistent decoder's plane holds, of
order 16 and others, at the ranks with rows of their own, with and without dense
corrections: the field equals the oracle decoder's."""
import numpy as np
import pytest

from test_gpu_decode_paths import _built, _check, _field  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cap", [1, 2, 3, 4, 5, 9])
@pytest.mark.parametrize("dims,block", [((40, 33, 17, 18), (32, 32, 16, 16)), ((64, 48, 8, 16), (64, 48, 4, 16)), ((96, 64, 16, 15), (96, 64, 16, 15))])
@pytest.mark.parametrize("rel", [2e-1, 1e-2, 1e-4])
def test_large(dims, block, cap, rel):
    f = _field(dims, 11, 0.01)
    _check(f, dims, block, rel * float(np.ptp(f)), cap, 0)
