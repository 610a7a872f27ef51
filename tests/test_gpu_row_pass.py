"""The encode kernel's row pass over block shapes (whole and partial lines,
columns that do and do not start on a bitmap word, every padded order), bounds
and correction sizes: each record replays through the oracle, and the stream
is the one the bisection writes."""
import numpy as np
import pytest
import torch

import oracle
from oracle import replay
from paper_2601_20113_gb300 import dls

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    oracle.build()


def _field(dims, seed, spikes=0.0):
    nx, ny, nz, nt = dims
    r = np.random.default_rng(seed)
    t, z, y, x = np.meshgrid(*[np.arange(n) / 16.0 for n in (nt, nz, ny, nx)], indexing="ij")
    f = np.zeros((nt, nz, ny, nx))
    for _ in range(6):
        k = r.uniform(0.2, 2.0, 4)
        f += np.sin(k[0] * t + k[1] * z + k[2] * y + k[3] * x + r.uniform(0, 6.28))
    f += 1e-3 * r.standard_normal(f.shape)
    f += spikes * r.standard_normal(f.shape) * (r.uniform(size=f.shape) < 0.01)
    return f[None].astype(np.float32)


def _stream(fd, block, eb, eb_type, cap, rank_mode):
    return dls.compress(fd, block=block, eb=eb, eb_type=eb_type, rank_cap=cap, precision=dls.PREC_FP32,
                        rank_mode=rank_mode).cpu().numpy().copy()


def _check(f, dims, block, eb, eb_type=dls.EB_ABS, cap=16):
    fd = torch.from_numpy(f).cuda()
    tail = _stream(fd, block, eb, eb_type, cap, dls.RANK_TAIL)
    search = _stream(fd, block, eb, eb_type, cap, dls.RANK_SEARCH)
    cfg = oracle.Config(dims, block, oracle.F32, eb=eb, eb_type=eb_type, rank_cap=cap)
    res, errs = replay.replay_stream(cfg, f, tail)
    bad = [r["errors"] for r in res if r["errors"]]
    assert not errs and not bad, (errs, bad[:3])
    tail[67] = search[67] = 0                          # header byte: rank mode used
    assert tail.size == search.size and np.array_equal(tail, search)


SHAPES = [((32, 32, 16, 32), (16, 16, 16, 16)),        # the common block
          ((26, 21, 18, 18), (16, 16, 16, 16)),        # partial lines, odd planes, two time steps
          ((35, 16, 9, 25), (16, 16, 8, 16)),          # unaligned lines, nine time steps
          ((32, 16, 8, 16), (8, 8, 8, 8)),             # order 8
          ((40, 20, 10, 12), (12, 8, 4, 4)),           # order 4
          ((39, 27, 5, 21), (13, 9, 5, 7)),            # odd everything, order 7
          ((64, 40, 3, 16), (32, 32, 1, 16)),          # several chunks a plane
          ((40, 34, 4, 16), (20, 17, 4, 16)),          # ... that do not tile it
          ((16, 8, 4, 33), (16, 8, 4, 11)),
          ((64, 48, 9, 20), (64, 48, 6, 16)),          # more points than the bitmap in shared memory holds
          ((30, 22, 13, 4), (30, 22, 13, 3))]


@pytest.mark.parametrize("dims,block", SHAPES)
@pytest.mark.parametrize("rel", [1e-2, 1e-3, 1e-4])
def test_shapes(dims, block, rel):
    f = _field(dims, 3)
    _check(f, dims, block, rel * float(np.ptp(f)))


@pytest.mark.parametrize("dims,block", SHAPES)
@pytest.mark.parametrize("eps", [0.05, 1.0])
def test_shapes_nrmse(dims, block, eps):
    _check(_field(dims, 4), dims, block, eps, dls.EB_NRMSE)


@pytest.mark.parametrize("spikes", [0.05, 0.5, 20.0, 1e5])
@pytest.mark.parametrize("cap", [2, 16])
def test_correction_sizes(spikes, cap):
    """Past |k| = 59, past a byte, escapes."""
    dims = (26, 21, 17, 18)
    _check(_field(dims, 5, spikes), dims, (16, 16, 16, 16), 2e-3, cap=cap)


def test_values_on_ties():
    dims = (32, 16, 16, 16)
    f = (np.round(_field(dims, 6) * 8) / 8).astype(np.float32)
    _check(f, dims, (16, 16, 16, 16), 0.125)
    _check(f, dims, (16, 16, 16, 16), 0.0625)
