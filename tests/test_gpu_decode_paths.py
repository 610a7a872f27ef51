"""The decoder over ranks, correction forms and widths, row alignments and
record sizes, where its paths change: the field equals the oracle decoder's."""
import numpy as np
import pytest
import torch

import oracle
from paper_2601_20113_gb300 import dls

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    oracle.build()


def _field(dims, seed, noise, dtype=np.float32):
    nx, ny, nz, nt = dims
    r = np.random.default_rng(seed)
    t, z, y, x = np.meshgrid(*[np.arange(n) / 16.0 for n in (nt, nz, ny, nx)], indexing="ij")
    f = np.zeros((nt, nz, ny, nx))
    for _ in range(9):
        k = r.uniform(0.2, 2.5, 4)
        f += np.sin(k[0] * t + k[1] * z + k[2] * y + k[3] * x + r.uniform(0, 6.28))
    f += noise * r.standard_normal(f.shape) * (r.uniform(size=f.shape) < 0.2)
    return f[None].astype(dtype)


def _check(f, dims, block, eb, rank_cap, codec, misalign=0):
    p = dls.make_params((1, dims[3], dims[2], dims[1], dims[0]), torch.float32, block, eb, dls.EB_ABS, rank_cap, corr_codec=codec)
    fd = torch.from_numpy(f).cuda()
    out = torch.empty(dls.compress_bound(p), dtype=torch.uint8, device="cuda")
    ws = torch.empty(dls.workspace_size(p), dtype=torch.uint8, device="cuda")
    st, nb = dls.compress_into(p, fd, out, ws)
    assert st == dls.OK
    base = torch.full((f.size + misalign,), float("nan"), device="cuda")
    got = base[misalign:].view(fd.shape)
    assert dls.decompress_into(out[:nb], got) == dls.OK
    st, ref = oracle.decompress(out[:nb].cpu().numpy())
    assert st == 0 and np.array_equal(got.cpu().numpy(), ref)


B16 = (16, 16, 16, 16)
DIMS = (36, 20, 17, 19)            # edges of 4, 4, 1 and 3: aligned lines


@pytest.mark.parametrize("rank_cap", [0, 1, 2, 3, 4, 5, 7, 8, 9, 16])
@pytest.mark.parametrize("codec", [0, 1])
def test_ranks(rank_cap, codec):
    f = _field(DIMS, 5, 0.0)
    _check(f, DIMS, B16, 2e-3 * float(np.ptp(f)), rank_cap, codec)


# noise in steps of the bound: correction widths from 1 bit to past the nibble and past 8 bits, escapes at the last
@pytest.mark.parametrize("steps", [0.6, 1.5, 3, 7, 20, 120, 4e6])
@pytest.mark.parametrize("codec", [0, 1])
@pytest.mark.parametrize("dims", [DIMS, (37, 18, 16, 16)])
def test_correction_widths(steps, codec, dims):
    eb = 2e-3
    _check(_field(dims, 6, 2 * eb * steps), dims, B16, eb, 5, codec)


@pytest.mark.parametrize("dims,block,misalign", [((32, 16, 16, 16), B16, 1), ((34, 16, 16, 16), B16, 0), ((30, 14, 8, 12), (10, 7, 8, 6), 0),
                                                 ((24, 8, 8, 32), (4, 2, 1, 16), 0), ((9, 5, 3, 20), (2, 2, 1, 10), 0),
                                                 ((64, 64, 2, 8), (64, 64, 2, 8), 0), ((65, 64, 2, 8), (65, 64, 2, 8), 0)])
@pytest.mark.parametrize("codec", [0, 1])
def test_shapes(dims, block, misalign, codec):
    f = _field(dims, 7, 0.01)
    _check(f, dims, block, 1e-3 * float(np.ptp(f)), 8, codec, misalign)


def test_records_beyond_the_stage():
    """White noise: wide columns, dense corrections and raw blocks of every size class."""
    r = np.random.default_rng(8)
    f = r.standard_normal((1, 32, 16, 32, 32)).astype(np.float32)
    for eb in (0.3, 0.03, 3e-3, 1e-6):
        for cap in (1, 4, 8):
            _check(f, (32, 32, 16, 32), B16, eb, cap, 1)
