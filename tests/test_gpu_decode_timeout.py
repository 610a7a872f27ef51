"""A record whose copy never arrives: the decoder's bounded wait runs out, the
call returns the timeout, and the next call is whole."""
import numpy as np
import pytest
import torch

from paper_2601_20113_gb300 import dls, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("block", [0, 5])
def test_withheld_record(block):
    f = synth.modes3d(32, 32, 32, 32, seed=2, device="cuda")
    comp = dls.compress(f, (16, 16, 16, 16), 1e-3 * float(f.max() - f.min()))
    ref, out = dls.decompress(comp).cpu().numpy(), torch.empty_like(f)
    assert dls.set_fault_hook(dls.FAULT_WITHHOLD_RECORD, block) == dls.OK
    try:
        st = dls.decompress_into(comp, out)
    finally:
        assert dls.set_fault_hook(dls.FAULT_NONE) == dls.OK
    assert st == dls.ERR_TIMEOUT, dls.status_string(st)
    torch.cuda.synchronize()
    assert dls.decompress_into(comp, out) == dls.OK and np.array_equal(out.cpu().numpy(), ref)
