"""mhd_get_state returns only when the buffers of earlier asynchronous gets are filled, on every path
it has (host in one piece or by slabs, device) and in every precision: the buffers are read with no
mhd_synchronize in between, the last value to arrive first."""
import numpy as np
import pytest
import torch

from paper_1810_12707_gb300 import mhd

pytestmark = pytest.mark.gpu


def buffers(n):
    pin = [torch.full(s, float("nan"), dtype=torch.float64).pin_memory() for s in ((n, n, n), (3, n, n, n), (3, n, n, n))]
    return pin, [p.numpy() for p in pin]


@pytest.mark.parametrize("device", [False, True])
@pytest.mark.parametrize("precision", [mhd.MHD_FP64, mhd.MHD_FP64_DF, mhd.MHD_FP32_MIXED])
@pytest.mark.parametrize("n", [32, 128, 256])
def test_get_waits_for_an_asynchronous_get(n, precision, device):
    ctx = mhd.mhd_init(n, [(1e-2, 1e-2, 10.0)] * 2, precision=precision)
    gen = torch.Generator("cuda").manual_seed(n)
    fields = [torch.randn(s, dtype=torch.float64, device="cuda", generator=gen) for s in ((n, n, n), (3, n, n, n), (3, n, n, n))]
    for i in range(2):
        mhd.mhd_set_state(ctx, i, *[f + i for f in fields])
    keep, out = buffers(n)
    mhd.mhd_get_state_async(ctx, 0, *out)
    other = mhd.mhd_get_state(ctx, 1, device=device)
    last = out[2][2, -1, -1, -1]
    got = [a.copy() for a in out]
    assert last == last
    assert mhd.mhd_synchronize(ctx) == mhd.MHD_OK
    for g, a in zip(got, out):
        assert np.array_equal(g, a)
    ref = mhd.mhd_get_state(ctx, 0)
    for g, r in zip(got, ref):
        assert np.array_equal(g, r)
    assert not np.array_equal(got[0], other[0].cpu().numpy() if device else other[0])
    # the same buffers again: the second get's values are the ones that stay
    mhd.mhd_get_state_async(ctx, 0, *out)
    lib = mhd.load_library()
    assert lib.mhd_get_state(ctx.handle, 1, *[a.ctypes.data for a in out], 0) == mhd.MHD_OK
    got = [a.copy() for a in out]
    assert mhd.mhd_synchronize(ctx) == mhd.MHD_OK
    for g, r in zip(got, mhd.mhd_get_state(ctx, 1)):
        assert np.array_equal(g, r)
    mhd.mhd_destroy(ctx)
    del keep
