"""Which copies out to the device a kernel takes, compiled for the host: large ones
only where both addresses let it move 16 bytes at a time.  Runs without a GPU."""
import ctypes
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
SRC = os.path.join(HERE, "host_harness", "host_copy.cu")
MB = 1 << 20


@pytest.fixture(scope="module")
def hx(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    out = str(tmp_path_factory.mktemp("hx") / "libhostcopy.so")
    subprocess.check_call([nvcc, "-O2", "-std=c++17", "-Xcompiler", "-fPIC", "-shared",
                           "-gencode", "arch=compute_103a,code=sm_103a", "-o", out, SRC,
                           "-I", os.path.join(HERE, "..", "include")])
    L = ctypes.CDLL(out)
    L.hx_copy_by_kernel.argtypes = [ctypes.c_ulonglong] * 3
    return L


@pytest.mark.parametrize("dst,src,most", [(0, 0, 64), (16, 4096, 64), (1, 0, 8), (4, 0, 8), (8, 16, 8),
                                          (0, 2, 8), (3, 3, 8)])
def test_limits(hx, dst, src, most):
    base = 1 << 40
    for d in (-1, 0, 1):
        assert hx.hx_copy_by_kernel(base + dst, base + src, most * MB + d) == (d <= 0)
    assert hx.hx_copy_by_kernel(base + dst, base + src, 0) == 1
