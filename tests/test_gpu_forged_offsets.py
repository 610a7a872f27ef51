"""Offset tables with entries near 2^64, whose sums with the payload's position
wrap: the decoders refuse the records, the verification leaves them out."""
import numpy as np
import pytest
import torch

from paper_2601_20113_gb300 import dls, synth

pytestmark = pytest.mark.gpu

TOP = 1 << 64
# (entry k, entry k + 1)
FORGED = [(TOP - 4096, TOP - 16), (1 << 63, TOP - 16), (TOP - 80000, TOP - 128), (TOP - 16, 64), (TOP - 32, 0), (TOP - 32, TOP - 16)]


def _forge(comp, at, k, pair):
    s = comp.cpu().numpy().copy()
    table = s[at + 8 * k:at + 8 * k + 16].view(np.uint64)
    table[:] = np.array(pair, np.uint64)
    return torch.from_numpy(s).cuda()


@pytest.mark.parametrize("pair", FORGED)
@pytest.mark.parametrize("dtype,block", [(torch.float32, (16, 16, 16, 16)), (torch.float32, (8, 8, 8, 32)), (torch.float32, (4, 2, 1, 16)),
                                         (torch.float64, (16, 16, 16, 16))])
def test_block_streams(dtype, block, pair):
    f = synth.modes3d(32, 32, 32, 32, seed=2, device="cuda").to(dtype)
    comp = dls.compress(f, block, 1e-2 * float(f.max() - f.min()))
    at = 128 + 32                                   # header, one variable's record
    nb = dls.stream_info(comp).total_blocks
    for k in (0, 1, nb // 2, nb - 1):
        bad = _forge(comp, at, k, pair)
        assert dls.decompress_into(bad, torch.empty_like(f)) == dls.ERR_CORRUPT
        rep, good = dls.verify(f, f, bad), dls.verify(f, f, comp)
        assert rep["sum_sq_err"] == 0 and rep["n_corr"] <= good["n_corr"] and rep["mean_rank"] < good["mean_rank"]


@pytest.mark.parametrize("pair", FORGED)
def test_global_streams(pair):
    f = synth.modes3d(16, 16, 16, 4, seed=2, device="cuda")[0].contiguous()
    comp = dls.gb_compress(f, 4, 1.0, synth.patch_origins((16, 16, 16), (4, 4, 4), 256, seed=1))
    at, nrec = 80 + 8 * 64 * 64, 4 * 64
    for k in (1, nrec // 2, nrec - 2):
        out = torch.empty(f.shape, dtype=torch.float64, device="cuda")
        assert dls.gb_decompress_into(_forge(comp, at, k, pair), out) == dls.ERR_CORRUPT
