"""The FP64 reciprocal, quotient and square root that the kernels use in place of divisions and library
roots (csrc/fp64_util.cuh), against exact rational arithmetic.

Bounds, in units in the last place of the result: each rounds once, in its last fused multiply-add
(1/2).  The reciprocal and the root add their iteration's remaining error, below 2^-57 relative, which is
below 2^-4 units; the quotient adds its remainder's product with the error of the reciprocal, below
2^-50 units.
"""
import ctypes
import math
import os
import shutil
import subprocess
from fractions import Fraction

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1810_12707_gb300", "csrc")
NVCC = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
RCP, QUOTIENT, SQRT, COVERS, RCP_ANY = range(5)


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("fp64_util") / "probe.so")
    subprocess.check_call([NVCC, "-O3", "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", "-shared",
                           "-Xcompiler", "-fPIC", "-I", CSRC, os.path.join(ROOT, "tests", "fp64_util_probe.cu"),
                           "-o", out])
    lib = ctypes.CDLL(out)

    def call(which, a, b=None):
        a = np.ascontiguousarray(a, dtype=np.float64)
        b = a if b is None else np.ascontiguousarray(b, dtype=np.float64)
        r = np.empty_like(a)
        assert lib.fp64_util_probe(which, len(a), *[ctypes.c_void_p(x.ctypes.data) for x in (a, b, r)]) == 0
        return r

    return call


def numbers(seed, count, lo, hi):
    """Random mantissas (some with long runs of zeros or ones), exponents from lo to hi, both signs."""
    rng = np.random.default_rng(seed)
    m = rng.integers(0, 2 ** 52, count)
    m[::7] &= ~((1 << 40) - 1)
    m[1::7] |= (1 << 40) - 1
    m[2::53], m[3::53] = 0, 2 ** 52 - 1
    x = np.ldexp(1.0 + m / 2.0 ** 52, rng.integers(lo, hi + 1, count))
    return np.where(rng.random(count) < 0.5, x, -x)


def ulps(value, exact):
    """|value - exact| in units in the last place of the exact result."""
    return abs(Fraction(float(value)) - exact) / Fraction(math.ulp(float(exact)))


@pytest.mark.parametrize("which", [RCP, RCP_ANY])
def test_reciprocal(run, which):
    x = np.concatenate([numbers(1, 12000, -1021, 1020), numbers(2, 4000, -3, 3),
                        [2.0 ** -1021, -2.0 ** -1021, np.nextafter(2.0 ** 1021, 0)]])
    r = run(which, x)
    assert max(ulps(v, 1 / Fraction(float(a))) for v, a in zip(r, x)) <= 0.5 + 2.0 ** -4


def test_quotient(run):
    x = np.concatenate([numbers(3, 12000, -500, 500), numbers(4, 4000, -1, 1), numbers(5, 2000, -1021, -900),
                        numbers(6, 2000, 900, 1020)])
    m = np.concatenate([numbers(7, 12000, -500, 500), numbers(8, 4000, -1, 1), numbers(9, 2000, -940, 0),
                        numbers(10, 2000, 0, 1023)])
    q = run(QUOTIENT, m, x)
    assert max(ulps(v, Fraction(float(a)) / Fraction(float(b))) for v, a, b in zip(q, m, x)) <= 0.5 + 2.0 ** -10


def test_quotient_outside_the_range(run):
    x = np.array([2.0 ** -600, -2.0 ** -600, 0.3, -0.3, 0.3, 1.7, 1.7, 2.0 ** 900])
    m = np.array([2.0 ** 600, 2.0 ** 600, np.inf, np.inf, -np.inf, np.nan, 0.0, 2.0 ** -900])
    q = run(QUOTIENT, m, x)
    with np.errstate(all="ignore"):
        assert np.array_equal(q, m / x, equal_nan=True)


def test_square_root(run):
    x = np.abs(np.concatenate([numbers(11, 12000, -1022, 1023), numbers(12, 4000, -2, 2),
                               [2.0 ** -1022, 2.0 ** -959, np.nextafter(2.0 ** -959, 0), np.finfo(float).max]]))
    r = run(SQRT, x)

    def error(v, a):
        # the root to 2^-40 units: an integer root of a 2^(2 s), s so that it has 93 bits or more
        s = 93 - math.frexp(a)[1] // 2
        f = Fraction(a) * Fraction(2) ** (2 * s)
        return ulps(v, Fraction(math.isqrt(f.numerator // f.denominator)) / Fraction(2) ** s)

    assert max(error(float(v), float(a)) for v, a in zip(r, x)) <= 0.5 + 2.0 ** -4
    special = np.array([0.0, -0.0, 5e-324, 1e-310, -1.0, np.inf, -np.inf, np.nan])
    with np.errstate(all="ignore"):
        assert np.array_equal(run(SQRT, special), np.sqrt(special), equal_nan=True)


def test_the_range_of_the_reciprocal(run):
    edges = np.array([2.0 ** -1021, 2.0 ** 1021])
    x = np.concatenate([np.nextafter(edges, 0), edges, np.nextafter(edges, np.inf), [0.0, np.inf, np.nan, 5e-324, 1.0]])
    x = np.concatenate([x, -x])
    expected = (np.abs(x) >= edges[0]) & (np.abs(x) < edges[1])
    assert np.array_equal(run(COVERS, x) == 1.0, expected)
    with np.errstate(all="ignore"):  # outside it the general reciprocal divides
        assert np.array_equal(run(RCP_ANY, x[~expected]), 1.0 / x[~expected], equal_nan=True)
