"""The closed form of Euclidean rows (hd_euclid.cuh), compiled for the host: every
row it calls certain equals the exact search, no row with voxels is missed, and
few rows are left open, on scans of the usual shape, nearly axis-parallel paths,
strips of the major axis, radii on the voxel grid, and extreme geometries.  Runs
without a GPU."""
import ctypes
import math
import os
import shutil
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
SRC = os.path.join(HERE, "host_harness", "host_slice_rows.cu")


@pytest.fixture(scope="module")
def hx(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    out = str(tmp_path_factory.mktemp("hx") / "libhostrows.so")
    subprocess.check_call([nvcc, "-O2", "-std=c++17", "-Xcompiler", "-fPIC", "-shared",
                           "-Xcompiler", "-ffp-contract=off",
                           "-gencode", "arch=compute_103a,code=sm_103a",
                           "-diag-suppress", "20014", "-o", out, SRC,
                           "-I", os.path.join(HERE, "..", "include")])
    L = ctypes.CDLL(out)
    L.hx_slice_rows.restype = ctypes.c_longlong
    return L


@pytest.mark.parametrize("dims,vox,T,sigma,d0s", [
    ((64, 64, 8), (1.0, 1.0, 2.5), 100.0, 2.0, (0.5, 1.0, 2.5)),
    ((50, 41, 12), (0.93, 1.1, 1.9), 60.0, 0.5, (0.95, 3.3)),
    ((9, 70, 5), (1.0, 1.0, 1.0), 80.0, 4.0, (0.25, 1.5)),
    ((24, 24, 24), (1 / 64, 1 / 64, 1 / 64), 1.0, 0.01, (1 / 65536, 0.02)),
    ((12, 12, 9), (64.0, 64.0, 64.0), 4000.0, 60.0, (20.0, 64.0)),
    ((40, 30, 6), (1.0, 1.0, 1.0), 12.0, 3.0, (1.0,)),  # trackers inside the grid: not closed
])
def test_certain_rows_are_exact(hx, dims, vox, T, sigma, d0s):
    rng = np.random.default_rng(sum(dims))
    half = math.hypot(dims[0] * vox[0], dims[1] * vox[1]) / 2
    hz = dims[2] * vox[2] / 2
    total = left = 0
    for i in range(400):
        phi = math.radians(rng.choice([0.0, 90.0, 45.0, 4.0, 184.0, rng.uniform(0, 360)]))
        c, s = math.cos(phi), math.sin(phi)
        u0, v0 = rng.uniform(-half, half) * 1.05, rng.uniform(-hz, hz) * 1.2
        if i % 7 == 0:  # along a line of voxel centres
            u0, v0 = (0.5 + rng.integers(-3, 3)) * vox[1], (0.5 + rng.integers(-2, 2)) * vox[2]
        u1, v1 = (u0, v0) if i % 5 == 0 else (u0 + rng.normal(0, sigma), v0 + rng.normal(0, sigma))
        W = [-T * c - u0 * s, -T * s + u0 * c, v0, T * c - u1 * s, T * s + u1 * c, v1]
        W = (ctypes.c_longlong * 6)(*[int(round(x * 65536)) for x in W])
        for d0 in d0s:
            for m0, ln in ((0, max(dims)), (dims[1] // 3, max(1, dims[1] // 2))):
                opened, closed = ctypes.c_longlong(0), ctypes.c_int(0)
                n = hx.hx_slice_rows(W, *dims, *[ctypes.c_float(v) for v in vox], ctypes.c_float(T),
                                     ctypes.c_float(d0), m0, ln, ctypes.byref(opened),
                                     ctypes.byref(closed))
                assert n >= 0, (n, list(W), d0, m0)
                total += n
                left += opened.value
    if T > half * 1.1:
        assert total > 1000 and left < 0.2 * total
