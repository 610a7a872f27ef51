"""The lossless stage's two writers: values of up to a byte through a buffer,
wider ones directly; sparse and dense chunks, records that end inside one."""
import numpy as np
import pytest
import torch

import oracle
from oracle import replay
from paper_2601_20113_gb300 import dls, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    oracle.build()


# corrections of 2, 8, 9, 10 and 16 bits; entry lists and dense fields, and records where neither wins
@pytest.mark.parametrize("k", [1, 90, 160, 400, 20000])
@pytest.mark.parametrize("density", [0.0005, 0.01, 0.12, 0.4, 0.7])
@pytest.mark.parametrize("dims,block", [((40, 36, 20, 36), (16, 16, 8, 16)), ((27, 9, 7, 11), (9, 9, 7, 11))])
def test_stream_equals_the_oracles(k, density, dims, block):
    r = np.random.default_rng(7)
    f = synth.modes3d(*dims, seed=9, count=4).numpy()
    eb = 2e-3 * float(np.ptp(f))
    hit = r.uniform(size=f.shape) < density
    f = (f + np.where(hit, 2.0 * eb * r.uniform(-k, k, f.shape), 0.0)).astype(f.dtype)
    p = dls.make_params(f.shape, torch.float32, block, eb, dls.EB_ABS, 2, precision=dls.PREC_FP64,
                        rank_mode=dls.RANK_SEARCH, corr_codec=1)
    out = torch.empty(dls.compress_bound(p), dtype=torch.uint8, device="cuda")
    ws = torch.empty(dls.workspace_size(p), dtype=torch.uint8, device="cuda")
    st, nb = dls.compress_into(p, torch.from_numpy(f).cuda(), out, ws)
    assert st == dls.OK
    got = out[:nb].cpu().numpy()
    st, ref, _ = oracle.compress(oracle.Config(dims, block, oracle.F32, eb=eb, rank_cap=2, corr_codec=1), f)
    assert st == oracle.OK
    assert got.size == ref.size and np.array_equal(got, ref)
