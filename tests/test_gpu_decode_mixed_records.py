"""Records of every class of the float32 decoder in turn on the same CTA: listed
and Rice-coded corrections, dense ones whose records reach over the plane,
records that the general path stages itself, raw blocks, rank 0.  Several
blocks a resident CTA, so that every class follows every other in its buffers;
the field equals the oracle decoder's."""
import numpy as np
import pytest
import torch

import oracle
from oracle import replay
from paper_2601_20113_gb300 import dls

pytestmark = pytest.mark.gpu

EB = 1e-3
KINDS = ["listed", "over_the_plane", "rank_12", "zero", "wide_list", "raw", "smooth", "dense_9", "dense_3", "rank_12_dense"]


def _block(kind, r):
    t, z, y, x = np.meshgrid(*[np.arange(16) / 16.0] * 4, indexing="ij")
    f = np.sin(2 * x + y + 3 * t) + np.cos(z - 2 * t + x)
    noise, where = r.standard_normal(f.shape), r.uniform(size=f.shape)
    if kind == "listed":
        f += 2.5 * EB * noise * (where < 0.02)
    elif kind == "over_the_plane":
        f += 14 * EB * noise
    elif kind == "rank_12":
        f = sum(np.sin(3 * k * t + r.uniform(0, 6)) * np.cos(k * x + y * r.uniform(0, 3)) / k for k in range(1, 15))
    elif kind == "zero":
        f *= 0
    elif kind == "wide_list":
        f += 60 * EB * noise * (where < 0.02)
    elif kind == "raw":
        f = 1e6 * noise
    elif kind == "dense_9":
        f += 300 * EB * noise
    elif kind == "dense_3":
        f += 2 * EB * noise
    elif kind == "rank_12_dense":
        f += 6 * EB * noise
        f += 5 * sum(np.sin(3 * k * t + r.uniform(0, 6)) * np.cos(k * x + y * r.uniform(0, 3)) / k for k in range(1, 15))
    return f


def _tile():
    r = np.random.default_rng(12)
    return np.concatenate([_block(k, r) for k in KINDS], axis=1)[None].astype(np.float32)     # along z


def _config(codec, nz=16 * len(KINDS), cap=16):
    return oracle.Config((16, 16, nz, 16), (16, 16, 16, 16), oracle.F32, eb=EB, rank_cap=cap, corr_codec=codec)


@pytest.mark.parametrize("codec", [0, 1])
@pytest.mark.parametrize("cap", [4, 16])
def test_alternating_records(codec, cap):
    oracle.build()
    f = _tile()
    st, s, _ = oracle.compress(_config(codec, cap=cap), f)
    assert st == 0
    st, ref = oracle.decompress(s)
    assert st == 0
    reps = 300                                   # 3000 blocks: six and a half a resident CTA
    big = torch.from_numpy(f).cuda().repeat(1, 1, reps, 1, 1)
    p = dls.make_params(tuple(big.shape), torch.float32, (16, 16, 16, 16), EB, dls.EB_ABS, cap, corr_codec=codec)
    out = torch.empty(dls.compress_bound(p), dtype=torch.uint8, device="cuda")
    ws = torch.empty(dls.workspace_size(p), dtype=torch.uint8, device="cuda")
    st, nb = dls.compress_into(p, big, out, ws)
    assert st == dls.OK
    want = torch.from_numpy(ref).cuda().repeat(1, 1, reps, 1, 1)
    got = torch.empty_like(big)
    for _ in range(3):
        got.fill_(float("nan"))
        assert dls.decompress_into(out[:nb], got) == dls.OK
        assert torch.equal(got, want)
