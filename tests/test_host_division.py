"""fdiv32, the division of the walk set-ups (hd_geom.cuh), compiled for the host: the
floor and the remainder over its whole range, at multiples of the divisor and one
beside them, for divisors up to 2^31 - 1 and quotients up to 2^20 of either sign.
Runs without a GPU."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
SRC = os.path.join(HERE, "host_harness", "host_division.cu")


@pytest.fixture(scope="module")
def hx(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    out = str(tmp_path_factory.mktemp("hx") / "libhostdivision.so")
    subprocess.check_call([nvcc, "-O2", "-std=c++17", "-Xcompiler", "-fPIC", "-shared",
                           "-gencode", "arch=compute_103a,code=sm_103a",
                           "-diag-suppress", "20014", "-o", out, SRC,
                           "-I", os.path.join(HERE, "..", "include")])
    L = ctypes.CDLL(out)
    L.hx_fdiv32.argtypes = [ctypes.c_longlong, ctypes.c_int, ctypes.POINTER(ctypes.c_longlong)]
    return L


@pytest.mark.parametrize("bits", [1, 2, 8, 17, 24, 30, 31])
def test_floor_and_remainder(hx, bits):
    rng = np.random.default_rng(bits)
    rem = ctypes.c_longlong()
    for k in range(4000):
        b = 2 ** bits - 1 if k % 7 == 0 else int(rng.integers(2 ** (bits - 1), 2 ** bits))
        q = int(rng.integers(-2 ** 20 + 2, 2 ** 20 - 2)) if k % 3 else int(rng.choice(
            [-2 ** 20 + 2, -1, 0, 1, 2 ** 20 - 2]))
        for a in (q * b, q * b - 1, q * b + 1, q * b + b // 2):
            got = hx.hx_fdiv32(a, b, ctypes.byref(rem))
            assert (got, rem.value) == divmod(a, b), (a, b)
