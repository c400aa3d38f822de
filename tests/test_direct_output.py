"""Device outputs are stored into by a kernel only where the context's GPU may store doubles: its own
memory at a double's alignment.  Every other pointer that a copy can write to takes a copy."""
import ctypes
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1810_12707_gb300", "csrc")
NVCC = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
UNREGISTERED, HOST, DEVICE, MANAGED = range(4)  # enum cudaMemoryType


@pytest.fixture(scope="module")
def choice(tmp_path_factory):
    if not os.path.exists(NVCC):
        pytest.skip("no nvcc")
    out = str(tmp_path_factory.mktemp("direct") / "direct.so")
    subprocess.check_call([NVCC, "-O2", "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", "-shared",
                           "-Xcompiler", "-fPIC", "-I", CSRC, "-x", "cu",
                           os.path.join(ROOT, "tests", "direct_output_host.cpp"), "-o", out])
    fn = ctypes.CDLL(out).direct_output_choice
    fn.argtypes = [ctypes.c_int, ctypes.c_int, ctypes.c_int, ctypes.c_ulonglong]
    return fn


def test_only_aligned_memory_of_the_same_gpu_is_stored_into(choice):
    base = 0x7f0000000000
    for device in (0, 1, 3):
        assert choice(DEVICE, device, device, base) == 1
        assert choice(DEVICE, device, device, base + 8) == 1
        for offset in (1, 2, 4, 12):
            assert choice(DEVICE, device, device, base + offset) == 0
        assert choice(DEVICE, device + 1, device, base) == 0
        for kind in (UNREGISTERED, HOST, MANAGED):
            assert choice(kind, device, device, base) == 0
            assert choice(kind, -2, device, base) == 0
