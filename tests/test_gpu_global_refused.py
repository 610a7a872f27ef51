"""What the global-basis mode refuses inside its sample: non-finite values in a
sampled patch of the first snapshot, and origins outside it among good ones.
The call returns the status and later calls on the same workspace sizes work."""
import numpy as np
import pytest
import torch

from paper_2601_20113_gb300 import dls, synth
from test_gpu_global import _built, _check  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


def _status(f, m, origins):
    with pytest.raises(dls.DlsError) as e:
        dls.gb_compress(f, m, 1.0, origins)
    return e.value.status


@pytest.mark.parametrize("m", [3, 4, 5])
@pytest.mark.parametrize("value", [float("nan"), float("inf"), -float("inf")])
def test_non_finite_sample(m, value):
    n = 4 * m
    f = torch.from_numpy(synth.modes3d(n, n, n, 3, seed=3, count=8).numpy()[0]).cuda()
    origins = synth.patch_origins((n, n, n), (m, m, m), 4 * m ** 3, seed=4)
    x, y, z = (int(v) for v in origins[0])
    f[0, z + m - 1, y, x + 1] = value
    assert _status(f, m, origins) == -3
    f[0, z:z + m, y:y + m, x:x + m] = value              # the whole patch
    assert _status(f, m, origins) == -3
    f[0] = value                                         # every sample
    assert _status(f, m, origins) == -3


@pytest.mark.parametrize("m", [3, 4, 5])
def test_origins_outside_among_good_ones(m):
    n = 4 * m
    f = torch.from_numpy(synth.modes3d(n, n, n, 3, seed=5, count=8).numpy()[0]).cuda()
    good = synth.patch_origins((n, n, n), (m, m, m), 4 * m ** 3, seed=6)
    for row, bad in ((0, (n - m + 1, 0, 0)), (7, (0, -1, 0)), (len(good) - 1, (0, 0, n)), (3, (2 ** 40, 0, 0))):
        o = np.array(good)
        o[row] = bad
        assert _status(f, m, o) == -1
    assert _status(f, m, np.full_like(good, -1)) == -1    # none inside
    _check(f.cpu().numpy(), m, 1.0)                       # and the next call is whole
