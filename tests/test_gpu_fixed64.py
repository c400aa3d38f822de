"""The FP64 transforms on the GPU at every group shape of the pencil (part of a warp, one warp,
several), with fields of very different magnitudes in one state.

Bound: a forward and an inverse 3D transform are six passes, each within 2^-52 of its pencils' norm
(see test_fixed64.py), so the round trip of a field cut to the kept modes is within 6 * 2^-52
relative L2, and its spectrum within 3 * 2^-52 plus the reference transform's own 3 * 2^-52.
"""
import numpy as np
import pytest

from paper_1810_12707_gb300 import mhd

pytestmark = pytest.mark.gpu


def project(f):
    n = f.shape[-1]
    k1, kr = np.abs(np.fft.fftfreq(n, 1.0 / n)), np.fft.rfftfreq(n, 1.0 / n)
    keep = (3 * k1[:, None, None] < n) & (3 * k1[None, :, None] < n) & (3 * kr[None, None, :] < n)
    s = np.fft.rfftn(f) * keep
    return s / n ** 3, np.fft.irfftn(s, s=f.shape, axes=(0, 1, 2))


@pytest.mark.parametrize("n", [16, 32, 64, 128, 256])
def test_round_trip_over_magnitudes(n):
    rng = np.random.default_rng(n)
    rho = 1.0 + 0.1 * rng.standard_normal((n, n, n))
    u = rng.standard_normal((3, n, n, n))
    b = rng.standard_normal((3, n, n, n)) * np.array([1e-150, 1e-3, 1e150])[:, None, None, None]
    b[1, :, n // 2] *= 1e-40
    ctx = mhd.mhd_init(n, [(1e-2, 1e-2, 10.0)])
    mhd.mhd_set_state(ctx, 0, rho, u, b)
    got = mhd.mhd_get_state(ctx, 0)
    fields = [rho] + [rho * u[c] for c in range(3)] + [b[c] for c in range(3)]
    out = [got[0]] + list(got[1]) + list(got[2])
    for q, (f, g) in enumerate(zip(fields, out)):
        spec, ref = project(f / np.abs(f).max())
        s = np.abs(f).max()
        assert np.linalg.norm(g / s - ref) <= 12 * 2.0 ** -52 * np.linalg.norm(ref), q
        sp = mhd.mhd_get_spectrum(ctx, 0, q) / s
        assert np.linalg.norm(sp - spec) <= 6 * 2.0 ** -52 * np.linalg.norm(spec), q
    mhd.mhd_destroy(ctx)


def test_a_nan_stays_in_its_field():
    n = 32
    rng = np.random.default_rng(5)
    rho, u, b = np.ones((n, n, n)), rng.standard_normal((3, n, n, n)), rng.standard_normal((3, n, n, n))
    b[2, 3, 4, 5] = np.nan
    ctx = mhd.mhd_init(n, [(1e-2, 1e-2, 10.0)])
    mhd.mhd_set_state(ctx, 0, rho, u, b)
    r, m, bb = mhd.mhd_get_state(ctx, 0)
    assert np.isfinite(r).all() and np.isfinite(m).all() and np.isfinite(bb[:2]).all() and np.isnan(bb[2]).all()
    mhd.mhd_destroy(ctx)
