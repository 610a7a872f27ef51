"""Fields of subnormal values: a decoded value may underflow to a zero of
negative sign, which a correction of zero leaves as it is.  Bit for bit the
oracle decoder's field."""
import numpy as np
import pytest
import torch

import oracle
from paper_2601_20113_gb300 import dls

pytestmark = pytest.mark.gpu


# dense and listed corrections, whole lines of 16 bytes and not
@pytest.mark.parametrize("scale,eb", [(1e-43, 2e-44), (3e-43, 5e-44), (1e-42, 1e-43), (1e-44, 3e-45), (1e-43, 2e-43)])
@pytest.mark.parametrize("dims", [(32, 16, 16, 16), (29, 17, 16, 16)])
@pytest.mark.parametrize("cap", [2, 4])
@pytest.mark.parametrize("codec", [0, 1])
def test_bits(scale, eb, dims, cap, codec):
    oracle.build()
    nx, ny, nz, nt = dims
    r = np.random.default_rng(0)
    t, z, y, x = np.meshgrid(*[np.arange(n) / 16 for n in (nt, nz, ny, nx)], indexing="ij")
    f = (scale * (np.sin(3 * x + y + 3 * t) * np.cos(2 * z - t) + 0.2 * r.standard_normal(x.shape)))[None].astype(np.float32)
    st, s, _ = oracle.compress(oracle.Config(dims, (16, 16, 16, 16), oracle.F32, eb=eb, rank_cap=cap, corr_codec=codec), f)
    assert st == 0
    st, ref = oracle.decompress(s)
    assert st == 0
    got = torch.empty(f.shape, device="cuda")
    assert dls.decompress_into(torch.from_numpy(s).cuda(), got) == dls.OK
    assert np.array_equal(got.cpu().numpy().view(np.uint32), ref.view(np.uint32))
