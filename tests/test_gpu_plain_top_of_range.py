"""Float32 fields within a quantization step of the largest float, in the plain
form: a rank whose decode overflows to infinity fails its test, as in the
oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_2601_20113_gb300 import dls

pytestmark = pytest.mark.gpu

DIMS, BLOCK = (16, 16, 4, 16), (16, 16, 4, 16)


def _field(lo, hi, seed=0):
    r = np.random.default_rng(seed)
    return r.uniform(lo, hi, (1, DIMS[3], DIMS[2], DIMS[1], DIMS[0])).astype(np.float32)


@pytest.fixture(scope="module", autouse=True)
def _built():
    oracle.build()


@pytest.mark.parametrize("lo,hi", [(3.3966e38, 3.4e38), (3.2e38, 3.4e38), (-3.4e38, 3.4e38)])
@pytest.mark.parametrize("eb", [1.0, 0.1])
@pytest.mark.parametrize("block", [BLOCK, (16, 16, 4, 3), (3, 2, 1, 16)])
def test_nrmse(lo, hi, eb, block):
    """Blocks stored raw where no decode is finite; the header's bound and step
    come from a norm summed in another order, so they are compared as numbers."""
    f = _field(lo, hi)
    st, ref, _ = oracle.compress(oracle.Config(DIMS, block, oracle.F32, eb=eb, eb_type=oracle.EB_NRMSE, rank_cap=16), f)
    assert st == 0
    comp = dls.compress(torch.from_numpy(f).cuda(), block=block, eb=eb, eb_type=oracle.EB_NRMSE, rank_cap=16)
    got = comp.cpu().numpy()
    assert got[136:152].view(np.float64) == pytest.approx(ref[136:152].view(np.float64), rel=1e-12, abs=0)
    got[136:152] = ref[136:152]
    assert np.array_equal(got, ref)
    assert torch.isfinite(dls.decompress(comp)).all()


@pytest.mark.parametrize("lo,hi", [(3.3966e38, 3.4e38), (3.2e38, 3.4e38)])
@pytest.mark.parametrize("eb", [1e36, 2e34])
@pytest.mark.parametrize("block", [BLOCK, (16, 16, 4, 3), (3, 2, 1, 16)])
def test_pointwise(lo, hi, eb, block):
    f = _field(lo, hi)
    st, ref, _ = oracle.compress(oracle.Config(DIMS, block, oracle.F32, eb=eb, rank_cap=16), f)
    assert st == 0
    comp = dls.compress(torch.from_numpy(f).cuda(), block=block, eb=eb, rank_cap=16)
    assert np.array_equal(comp.cpu().numpy(), ref)
    assert np.abs(dls.decompress(comp).cpu().numpy().astype(np.float64) - f).max() <= eb
