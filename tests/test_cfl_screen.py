"""The flux pass's CFL screen on the host: a point whose speed |u| + sqrt(cs^2 + |B|^2 / rho) exceeds the
maximum published so far always has its exact speed formed, at every density (very large and very
small ones, negative ones), and one well below it at ordinary densities does not."""
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
    out = str(tmp_path_factory.mktemp("cfl") / "cfl.so")
    subprocess.check_call([NVCC, "-O2", "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", "-shared",
                           "-Xcompiler", "-fPIC", "-I", CSRC, "-x", "cu",
                           os.path.join(ROOT, "tests", "cfl_screen_host.cpp"), "-o", out])
    return ctypes.CDLL(out)


def points(decades, count=200_000, negative=False):
    """(ux, uy, uz, cs^2, |B|^2, 1/rho) with |B|^2 / rho and u of ordinary size, rho over 10^+-decades,
    and their speeds."""
    rng = np.random.default_rng(int(decades) + 7 * negative)
    rho = 10.0 ** rng.uniform(-decades, decades, count)
    cs2 = 10.0 ** rng.uniform(-6, 3, count)
    va2 = 10.0 ** rng.uniform(-6, 6, count)
    if negative:
        rho = -rho
        va2 = -cs2 * (1 - 10.0 ** rng.uniform(-7, 0, count))
    u = rng.standard_normal((count, 3)) * 10.0 ** rng.uniform(-4, 2, (count, 1))
    b2, ir = va2 * rho, 1.0 / rho
    s = np.sqrt((u * u).sum(1)) + np.sqrt(cs2 + b2 * ir)
    return np.ascontiguousarray(np.column_stack([u, cs2, b2, ir])), s


def need(lib, df, p, published):
    out = np.zeros(len(p), dtype=np.int32)
    pub = np.ascontiguousarray(published)
    lib.cfl_screen_points(df, len(p), *[ctypes.c_void_p(a.ctypes.data) for a in (p, pub, out)])
    return out.astype(bool)


@pytest.mark.parametrize("negative", [False, True])
@pytest.mark.parametrize("df,decades", [(0, 0.5), (0, 20), (0, 60), (0, 150), (1, 0.5), (1, 15)])
def test_a_point_above_the_published_maximum_is_never_screened(lib, df, decades, negative):
    p, s = points(decades, negative=negative)
    assert need(lib, df, p, s * (1 - 1e-7)).all()


@pytest.mark.parametrize("df", [0, 1])
def test_points_below_it_are_screened(lib, df):
    p, s = points(2)
    assert not need(lib, df, p, s * (1 + 1e-5)).any()
