"""FP64 transforms of values near the ends of the double range (below 2^-959, above 2^976), at every
group shape of the pencil: set, spectrum and get of a field scaled by a power of two are those of the
unscaled field, scaled.

Bound: both runs are within 12 * 2^-52 of the exact round trip (6 * 2^-52 for a spectrum) in relative L2
(see test_gpu_fixed64.py), so within twice that of each other; the small fields' values are also
rounded to multiples of 2^-1074: 2^-69 of fields at 2^-1005, 2^-57 of their spectra at 2^-1017 (n = 256).
"""
import numpy as np
import pytest

from paper_1810_12707_gb300 import mhd

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [16, 32, 64, 128, 256])
def test_round_trip_near_the_ends_of_the_range(n):
    rng = np.random.default_rng(n)
    rho = 1.0 + 0.1 * rng.standard_normal((n, n, n))
    u, b = rng.standard_normal((3, n, n, n)), rng.standard_normal((3, n, n, n))
    powers = (-1005, -975, 985)
    ctx = mhd.mhd_init(n, [(1e-2, 1e-2, 10.0)] * 2)
    mhd.mhd_set_state(ctx, 0, rho, u, b)
    mhd.mhd_set_state(ctx, 1, rho, u, np.stack([np.ldexp(b[c], p) for c, p in enumerate(powers)]))
    for device in (False, True):
        one, two = mhd.mhd_get_state(ctx, 0, device=device), mhd.mhd_get_state(ctx, 1, device=device)
        if device:
            one, two = [t.cpu().numpy() for t in one], [t.cpu().numpy() for t in two]
        assert np.array_equal(one[0], two[0]) and np.array_equal(one[1], two[1])
        for c, p in enumerate(powers):
            assert np.linalg.norm(np.ldexp(two[2][c], -p) - one[2][c]) <= 24 * 2.0 ** -52 * np.linalg.norm(one[2][c]), p
    for c, p in enumerate(powers):
        s1, s2 = mhd.mhd_get_spectrum(ctx, 0, 4 + c), mhd.mhd_get_spectrum(ctx, 1, 4 + c)
        s2 = np.ldexp(s2.real, -p) + 1j * np.ldexp(s2.imag, -p)
        assert np.linalg.norm(s2 - s1) <= 12 * 2.0 ** -52 * np.linalg.norm(s1), p
    mhd.mhd_destroy(ctx)
