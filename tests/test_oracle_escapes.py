"""Blocks of escapes alone, whose records are larger than raw ones: the oracle
stores them raw."""
import numpy as np
import pytest

import oracle


@pytest.mark.parametrize("dtype,scale", [(oracle.F32, 3.4e38), (oracle.F64, 1.7e308)])
@pytest.mark.parametrize("block", [(16, 16, 4, 16), (16, 16, 4, 3), (3, 2, 1, 16)])
def test_stored_raw(dtype, scale, block):
    np_t = np.float32 if dtype == oracle.F32 else np.float64
    f = (scale * np.random.default_rng(0).uniform(0.999, 1.0, (1, 16, 4, 16, 16))).astype(np_t)
    eb = scale * 1e-18
    st, s, tr = oracle.compress(oracle.Config((16, 16, 4, 16), block, dtype, eb=eb, rank_cap=16), f, traces=True)
    assert st == oracle.OK and any(t.raw for t in tr)
    st, rec = oracle.decompress(s)
    assert st == oracle.OK and np.array_equal(rec[:, :], f)
