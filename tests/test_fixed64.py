"""The fixed-point arithmetic of the FP64 transforms (csrc/fixed64.cuh), compiled for the host and
compared with a discrete Fourier transform summed in long double.

Bounds: the result is rounded to FP64 once (relative error at most 2^-53 per value), and the
fixed-point stages add at most a unit per value and stage, each growing by sqrt(8) in the stages
that follow, where the unit is 2^-60 of the largest first-stage sum, in the worst of these inputs
(white noise, 1024 points) 2^-55 of the result's RMS: 2^-52 in all, in the L2 norm.
"""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1810_12707_gb300", "csrc")
NVCC = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    if not os.path.exists(NVCC):
        pytest.skip("no nvcc")
    out = str(tmp_path_factory.mktemp("fixed64") / "fixed64.so")
    subprocess.check_call([NVCC, "-O2", "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", "-shared",
                           "-Xcompiler", "-fPIC", "-I", CSRC, "-x", "cu", os.path.join(ROOT, "tests", "fixed64_host.cpp"),
                           os.path.join(CSRC, "twiddles.cu"), "-o", out])
    return ctypes.CDLL(out)


def transform(lib, x, direction, zp=0):
    y = np.array(x, dtype=np.complex128)
    lib.fixed64_fft(len(y), direction, zp, y.ctypes.data_as(ctypes.c_void_p))
    return y


def dft(x, direction):
    n = len(x)
    two_pi = 2 * np.arctan2(np.longdouble(0), np.longdouble(-1))
    j = np.arange(n)
    a = two_pi * direction * (np.outer(j, j) % n).astype(np.longdouble) / n
    c, s = np.cos(a), np.sin(a)
    xr, xi = x.real.astype(np.longdouble), x.imag.astype(np.longdouble)
    return c @ xr - s @ xi, s @ xr + c @ xi


def inputs(n):
    rng = np.random.default_rng(n)
    k = np.minimum(np.arange(n), n - np.arange(n))
    noise = rng.standard_normal(n) + 1j * rng.standard_normal(n)
    return {"noise": noise, "peak": np.where(k == 0, 1.0, 1e-3 * noise), "decay": np.exp(-0.5 * k) * noise,
            "row": (1 + 1e-9 * rng.standard_normal(n)).astype(complex), "single": np.where(np.arange(n) == n // 3, noise, 0),
            "small": 1e-250 * noise, "large": 1e250 * noise, "mixed": np.where(np.arange(n) % 5 == 0, 1e-30, 1.0) * noise}


@pytest.mark.parametrize("n", [16, 32, 64, 128, 256, 512, 1024])
def test_transform_matches_the_sum(lib, n):
    k = np.minimum(np.arange(n), n - np.arange(n))
    for name, x in inputs(n).items():
        for direction, zp in ((-1, 0), (+1, 0), (+1, 1)):
            z = np.where(3 * k < n, x, 0) if zp else x
            re, im = dft(z, direction)
            y = transform(lib, z, direction, zp)
            scale = np.sqrt(np.sum(re * re + im * im))
            if scale == 0:
                assert not y.any(), (name, direction, zp)
                continue
            err = float(np.sqrt(np.sum((y.real - re) ** 2 + (y.imag - im) ** 2)) / scale)
            assert err <= 2.0 ** -52, (name, direction, zp, err)


@pytest.mark.parametrize("n", [16, 128, 512])
def test_exact_and_exceptional_pencils(lib, n):
    for direction in (-1, +1):
        assert not transform(lib, np.zeros(n), direction).any()
        y = transform(lib, np.full(n, 0.3 - 1.7j), direction)  # sums of equal values are exact
        assert y[0] == n * (0.3 - 1.7j) and not y[1:].any()
        x = np.zeros(n, dtype=complex)
        x[0] = 0.1 + 2.3j
        assert np.array_equal(transform(lib, x, direction), np.full(n, 0.1 + 2.3j))
        for bad in (np.nan, np.inf, -np.inf):
            x = np.ones(n, dtype=complex)
            x[n // 2 + 1] = complex(0.0, bad)
            assert np.isnan(transform(lib, x, direction)).all()
        assert not transform(lib, np.full(n, 1e-300), direction).any()
