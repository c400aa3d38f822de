"""The set and get passes at every grid size and in every precision: device and host paths agree to
the bit, fields of one pencil block do not mix, and the diagnostics' own reciprocal and roots follow
the grid values over magnitudes.

Bound: the diagnostics are sums of up to 64^3 positive terms, each within a few units in the last
place, and FP64 sums of n terms in blocks round by less than 1e-14 relative; the fields they come
from are the transforms' (12 * 2^-52, see test_gpu_fixed64.py): 1e-13.
"""
import numpy as np
import pytest
import torch

from paper_1810_12707_gb300 import mhd

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [mhd.MHD_FP64, mhd.MHD_FP64_DF, mhd.MHD_FP32_MIXED])
@pytest.mark.parametrize("n", [16, 32, 64, 128])
def test_host_and_device_paths(n, precision):
    rng = np.random.default_rng(n)
    rho = 1.0 + 0.1 * rng.standard_normal((n, n, n))
    u, b = rng.standard_normal((3, n, n, n)), rng.standard_normal((3, n, n, n))
    u[1] = 0.0  # a field of zeros between others
    dev = [torch.from_numpy(a).cuda() for a in (rho, u, b)]
    ctx = mhd.mhd_init(n, [(1e-2, 1e-2, 10.0)] * 2, precision=precision)
    mhd.mhd_set_state(ctx, 0, rho, u, b)
    mhd.mhd_set_state(ctx, 1, *dev)
    assert np.array_equal(mhd.mhd_checkpoint(ctx, 0), mhd.mhd_checkpoint(ctx, 1))
    host, device = mhd.mhd_get_state(ctx, 0), mhd.mhd_get_state(ctx, 1, device=True)
    for h, g in zip(host, device):
        assert np.array_equal(h, g.cpu().numpy())
    assert not host[1][1].any()
    mhd.mhd_destroy(ctx)


@pytest.mark.parametrize("scale", [1e-160, 1e-3, 1.0, 1e100])
def test_diagnostics_over_magnitudes(scale):
    n = 64
    rng = np.random.default_rng(3)
    rho = np.full((n, n, n), 2.0)
    x = 2 * np.pi * np.arange(n) / n
    u = np.stack([np.cos((c + 1) * x)[None, None, :] * np.cos(2 * x)[:, None, None] + np.zeros((n, n, n)) for c in range(3)])
    b = scale * np.stack([np.sin((c + 2) * x)[None, :, None] + rng.uniform(1, 2) + np.zeros((n, n, n)) for c in range(3)])
    ctx = mhd.mhd_init(n, [(1e-2, 1e-2, 3.0)])
    mhd.mhd_set_state(ctx, 0, rho, u, b)
    d = mhd.mhd_diagnostics(ctx, 0)
    su, sb = np.sqrt((u * u).sum(0)), scale * np.sqrt(((b / scale) ** 2).sum(0))
    want = {"ke": np.mean(su * su), "mean_speed": np.mean(su), "mean_bmag": np.mean(sb), "eint": 9.0 * 2.0 * np.log(2.0)}
    if scale > 1e-100:
        want["me"] = 0.5 * np.mean(sb * sb)
        want["smax"] = np.max(su + np.sqrt(9.0 + sb * sb / 2.0))
    for k, v in want.items():
        if k == "mean_bmag" and scale < 1e-100:
            continue  # |B|^2 is below the FP64 range's normal numbers
        assert abs(d[k] - v) <= 1e-13 * abs(v), (k, d[k], v)
    mhd.mhd_destroy(ctx)
