"""How many path walks the system rows allocate where memory is short, compiled for
the host: as many as a chunk takes, or the most that halving finds, and none only
where not even the least fit.  Runs without a GPU."""
import ctypes
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
SRC = os.path.join(HERE, "host_harness", "host_rows_room.cu")
CHUNK, LEAST = 1 << 22, 1 << 10


@pytest.fixture(scope="module")
def hx(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    out = str(tmp_path_factory.mktemp("hx") / "libhostrowsroom.so")
    subprocess.check_call([nvcc, "-O2", "-std=c++17", "-Xcompiler", "-fPIC", "-shared",
                           "-gencode", "arch=compute_103a,code=sm_103a", "-o", out, SRC,
                           "-I", os.path.join(HERE, "..", "include")])
    L = ctypes.CDLL(out)
    L.hx_rows_room.restype = ctypes.c_longlong
    L.hx_rows_room.argtypes = [ctypes.c_longlong, ctypes.c_longlong, ctypes.POINTER(ctypes.c_int)]
    return L


@pytest.mark.parametrize("n", [1, 1000, LEAST, LEAST + 1, 5000, 1_800_000, CHUNK, CHUNK + 1, 1 << 32])
@pytest.mark.parametrize("room", [0, 1, LEAST - 1, LEAST, 3000, 1 << 20, CHUNK - 1, CHUNK, 1 << 40])
def test_room(hx, n, room):
    tries = ctypes.c_int()
    got = hx.hx_rows_room(n, room, ctypes.byref(tries))
    want = min(n, CHUNK)
    if room >= want:
        assert got == want and tries.value == 1
    elif room < min(want, LEAST):
        assert got == 0
    else:
        assert 0 < got <= room and (got == LEAST or 4 * got > room) and tries.value < 15
