"""The flux pass at exceptional densities: its reciprocal and its screened CFL speed.

A negative density with |B|^2 / |rho| > Cs^2 has no fast speed (a NaN), wherever in the grid it lies
and however low the flow's speed is there, so the screening must not skip it.  A density that
varies over sixteen decades tests the reciprocal: with m = rho u and u of order one, the products m u
and u x B are known, and the RHS of the induction equation, which holds u x B alone, is compared
with torch's FP64 transforms of the host's division.  Bound: the products are within 4 units in the
last place (2^-51 of |u||B|), the transforms within 6 * 2^-52 of the pencils' norms, and a
derivative scales both by at most k_max: 16 k_max 2^-52 of the largest |u x B|, in the L2 norm.
"""
import numpy as np
import pytest
import torch

from paper_1810_12707_gb300 import mhd

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [mhd.MHD_FP64, mhd.MHD_FP64_DF, mhd.MHD_FP32_MIXED])
@pytest.mark.parametrize("n", [16, 64])
def test_negative_density_stops_the_instance(n, precision):
    x = 2 * np.pi * np.arange(n) / n
    # one plane of negative density, band-limited so that it survives the 2/3 rule
    rho = 1.0 + 1.2 * np.cos(x)[None, None, :] * np.ones((n, n, 1))
    u = np.zeros((3, n, n, n))
    b = np.zeros((3, n, n, n))
    b[1] = 5.0
    ctx = mhd.mhd_init(n, [(1e-2, 1e-2, 1.0)], precision=precision)
    mhd.mhd_set_state(ctx, 0, rho, u, b)
    mhd.mhd_step(ctx, 1)
    assert mhd.mhd_synchronize(ctx) == mhd.MHD_ENONFINITE
    mhd.mhd_set_state(ctx, 0, np.abs(rho) + 0.5, u, b)
    mhd.mhd_step(ctx, 1)
    assert mhd.mhd_synchronize(ctx) == mhd.MHD_OK
    mhd.mhd_destroy(ctx)


def test_reciprocal_over_densities():
    n = 32
    rng = np.random.default_rng(9)
    for decade in range(-8, 9, 2):
        rho = 10.0 ** decade * (1.0 + 0.4 * np.cos(2 * np.pi * np.arange(n) / n))[None, None, :] * np.ones((n, n, 1))
        u0, b0 = rng.standard_normal((3, 1, n, 1)) * np.ones((3, n, n, n)), np.array([0.3, -0.7, 0.2])
        k1 = np.abs(np.fft.fftfreq(n, 1 / n))
        u0 = np.fft.ifft(np.fft.fft(u0, axis=2) * (k1 < 5)[None, None, :, None], axis=2).real  # rho u keeps inside the rule
        b = np.ones((3, n, n, n)) * b0[:, None, None, None]
        ctx = mhd.mhd_init(n, [(0.0, 0.0, 1.0)])
        mhd.mhd_set_state(ctx, 0, rho, u0, b)
        db = mhd.mhd_rhs(ctx, 0)[2]
        e = np.cross(u0, b0, axisa=0, axisb=0, axisc=0)
        kx = torch.fft.rfftfreq(n, 1 / n, dtype=torch.float64)[None, None, :]
        kk = torch.fft.fftfreq(n, 1 / n, dtype=torch.float64)
        k = [kx, kk[None, :, None], kk[:, None, None]]
        s = [torch.fft.rfftn(torch.from_numpy(np.ascontiguousarray(e[c]))) for c in range(3)]
        ref = [torch.fft.irfftn(1j * (k[(a + 1) % 3] * s[(a + 2) % 3] - k[(a + 2) % 3] * s[(a + 1) % 3]), s=(n, n, n))
               for a in range(3)]
        err = np.sqrt(sum(np.mean((db[a] - ref[a].numpy()) ** 2) for a in range(3)))
        assert err <= 16 * ((n - 1) // 3) * 2.0 ** -52 * np.abs(e).max(), (decade, err)
        mhd.mhd_destroy(ctx)
