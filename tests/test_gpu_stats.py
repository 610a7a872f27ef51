"""The statistics passes behind the range-relative and NRMSE bounds, at the
sizes where their loads change form: values exact, sums in the defined order."""
import numpy as np
import pytest
import torch

from paper_2601_20113_gb300 import dls

pytestmark = pytest.mark.gpu
CTAS, THREADS = 512, 256


def _field(shape, dtype, seed, offset=0):
    """A contiguous CUDA field whose first value lies `offset` values past an aligned address."""
    n = int(np.prod(shape))
    gen = torch.Generator(device="cuda").manual_seed(seed)
    base = torch.randn(n + offset, generator=gen, dtype=torch.float64, device="cuda").to(dtype)
    base[offset + n // 3] = 0.0
    base[offset + n // 2] = 1e-41 if dtype == torch.float32 else 1e-310      # subnormal
    return base[offset:].view(shape)


# K per variable: below one vector, off a multiple of it, and past a full unrolled step of a CTA's range
SHAPES = [(1, 2, 1, 3, 3), (2, 3, 1, 5, 7), (2, 4, 4, 8, 8), (1, 33, 17, 129, 31), (2, 48, 20, 64, 70)]


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("offset", [0, 1])
def test_relative_bound_is_the_exact_range(shape, dtype, offset):
    f = _field(shape, dtype, 5, offset)
    f[0].reshape(-1)[-1] = 7.5
    f[-1].reshape(-1)[0] = -6.25
    info = dls.stream_info(dls.compress(f, (2, 2, 1, 2), 1e-2, dls.EB_REL_RANGE))
    for v in range(shape[0]):
        assert info.eb[v] == 1e-2 * (f[v].max().double() - f[v].min().double()).item()


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("offset", [0, 1])
def test_sum_of_squares_keeps_its_order(shape, offset):
    f = _field(shape, torch.float32, 6, offset)
    p = dls.make_params(shape, torch.float32, (2, 2, 1, 2), 1.0, dls.EB_NRMSE)
    got = dls.field_stats(p, f)
    for v in range(shape[0]):
        x = f[v].cpu().numpy().astype(np.float64).ravel()
        per = -(-x.size // CTAS)
        steps = -(-per // THREADS)
        sq = np.zeros((CTAS, steps * THREADS))
        for c in range(CTAS):
            part = x[c * per:(c + 1) * per]
            sq[c, :part.size] = part * part              # exact: 24-bit factors
        s = np.zeros((CTAS, THREADS))
        for k in range(steps):
            s = s + sq[:, k * THREADS:(k + 1) * THREADS]
        o = THREADS // 2
        while o:
            s[:, :o] = s[:, :o] + s[:, o:2 * o]
            o //= 2
        total = 0.0
        for c in range(CTAS):
            total = total + s[c, 0]
        assert tuple(got[v]) == (x.min(), x.max(), total, x.size)


@pytest.mark.parametrize("bad", [float("nan"), float("inf"), -float("inf")])
@pytest.mark.parametrize("bound", [dls.EB_REL_RANGE, dls.EB_NRMSE])
@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
def test_non_finite_values_are_refused(bad, bound, dtype):
    f = _field((1, 16, 4, 20, 33), dtype, 7)
    f[0, 15, 3, 19, 32] = bad
    with pytest.raises(dls.DlsError) as e:
        dls.compress(f, (2, 2, 1, 2), 1e-2, bound)
    assert e.value.status == -3


@pytest.mark.parametrize("scale", [1e-38, 1e-40, 1e-44])
def test_subnormal_values_are_summed_exactly(scale):
    """Squares of subnormals, alone and beside the smallest normal values: sums of few terms, exact in any order."""
    shape = (1, 2, 1, 16, 300)
    f = torch.zeros(shape, dtype=torch.float32, device="cuda")
    flat = f.view(-1)
    vals = torch.tensor([scale, -3 * scale, 1.1754943508222875e-38, 0.0, -0.0], dtype=torch.float32)
    flat[::2000] = vals.cuda()
    p = dls.make_params(shape, torch.float32, (2, 2, 1, 2), 1.0, dls.EB_NRMSE)
    x = vals.numpy().astype(np.float64)
    got = dls.field_stats(p, f)[0]
    assert got[2] == pytest.approx(float(np.sum(x * x)), rel=5 * 2.0 ** -52)
