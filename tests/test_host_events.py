"""Event walks (hd_geom.cuh), compiled for the host, against the CPU oracle's
voxel sets: one update per change of row and two marks per walk decode to the
set itself and to the set dilated in-plane, on adversarial segments (ties,
planes, box edges) and generic ones.  Runs without a GPU."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

from tests.test_oracle_pins import _random_segments

HERE = os.path.dirname(os.path.abspath(__file__))
SRC = os.path.join(HERE, "host_harness", "host_events.cu")
I32P = ctypes.POINTER(ctypes.c_int32)


@pytest.fixture(scope="module")
def hx(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    out = str(tmp_path_factory.mktemp("hx") / "libhostevents.so")
    subprocess.check_call([nvcc, "-O2", "-std=c++17", "-Xcompiler", "-fPIC", "-shared",
                           "-gencode", "arch=compute_103a,code=sm_103a",
                           "-diag-suppress", "20014", "-o", out, SRC,
                           "-I", os.path.join(HERE, "..", "include")])
    return ctypes.CDLL(out)


def _generic(rng, n, dims):
    """Segments across the box in every direction, ends inside and outside."""
    d = np.array(dims)
    for _ in range(n):
        span = rng.choice([0.1, 1.0, 3.0])
        a = rng.uniform(-0.6, 1.6, 3) * d
        b = a + rng.uniform(-1.0, 1.0, 3) * d * span * np.array([1.0, 1.0, rng.choice([0.02, 1.0])])
        yield [np.round(65536 * v).astype(np.int32) for v in (a, b)]


def _dilate(v, dims, t):
    if t == 0 or v.size == 0:
        return np.sort(v)
    nx, ny, nz = dims
    vol = np.zeros((nz, ny, nx), bool)
    vol.reshape(-1)[v] = True
    out = vol.copy()
    for dy in range(-t, t + 1):
        for dx in range(-t, t + 1):
            s = vol[:, max(0, -dy):ny - max(0, dy), max(0, -dx):nx - max(0, dx)]
            if s.size:
                out[:, max(0, dy):ny - max(0, -dy), max(0, dx):nx - max(0, -dx)] |= s
    return np.flatnonzero(out.reshape(-1))


@pytest.mark.parametrize("dims,direct", [((5, 4, 1), 1), ((1, 1, 1), 1), ((1, 7, 1), 1),
                                         ((9, 1, 1), 1), ((40, 30, 1), 1), ((17, 64, 1), 1),
                                         ((12, 11, 3), 0), ((40, 30, 2), 0)])
def test_event_walks_equal_oracle(oracle_mod, hx, dims, direct):
    rng = np.random.default_rng(sum(dims) + 3)
    segs = list(_random_segments(rng, 1500, dims)) + list(_generic(rng, 1500, dims))
    seen = 0
    for a, b in segs:
        seg = np.concatenate([a, b]).astype(np.int32)
        ref = oracle_mod.voxel_set(np.asarray(a, np.int32), np.asarray(b, np.int32), *dims)
        for t in (0, 1, 3):
            if t and dims[2] > 1:
                continue
            out = np.zeros(int(np.prod(dims)), np.int32)
            runs = ctypes.c_int(0)
            n = hx.hx_events(seg.ctypes.data_as(I32P), *dims, t, direct, out.ctypes.data_as(I32P),
                             ctypes.byref(runs))
            if n == -1:
                continue
            assert n >= 0, (n, seg.tolist(), t)
            seen += n > 0
            assert np.array_equal(out[:n], _dilate(ref, dims, t)), (seg.tolist(), t)
    assert seen > 300


@pytest.mark.parametrize("dims", [(5, 4, 3), (1, 1, 1), (7, 1, 2), (40, 30, 20), (9, 1, 1),
                                  (64, 64, 8), (17, 200, 3)])
def test_path_walk_equals_run_walk(hx, dims):
    """Every run of the path walk is the general run walk's, in order; it
    declines only ties and paths without in-plane motion."""
    rng = np.random.default_rng(sum(dims) + 5)
    generic = list(_generic(rng, 4000, dims))
    taken = 0
    for k, (a, b) in enumerate(generic + list(_random_segments(rng, 4000, dims))):
        n = hx.hx_path(np.asarray(a, np.int32).ctypes.data_as(I32P),
                       np.asarray(b, np.int32).ctypes.data_as(I32P), *dims)
        assert n >= -1, (n, np.asarray(a).tolist(), np.asarray(b).tolist())
        taken += n >= 0 and k < len(generic)
    assert taken > 0.95 * len(generic)


@pytest.mark.parametrize("n,s", [(4096, 1 / 64), (128, 64.0), (4096, 2.0), (1, 64.0), (200, 1.0),
                                 (181, 0.93), (64, 0.015640259), (127, 63.99998)])
def test_grid_coordinate_is_exact(hx, n, s):
    """The two-product division of the world-to-grid map equals the floor over
    the whole range of world coordinates, at multiples of the voxel size too."""
    rng = np.random.default_rng(n)
    hx.hx_to_grid.restype = ctypes.c_longlong
    sq = int(round(s * 65536))
    w = np.concatenate([rng.integers(-2 ** 29, 2 ** 29, 200000), np.arange(-2 ** 29, -2 ** 29 + 99),
                        np.arange(2 ** 29 - 99, 2 ** 29), rng.integers(-2 ** 29 // sq, 2 ** 29 // sq,
                                                                       20000) * sq // 2])
    w = np.ascontiguousarray(w, dtype=np.int32)
    assert hx.hx_to_grid(n, ctypes.c_float(s), w.ctypes.data_as(I32P), ctypes.c_longlong(w.size)) == 0


@pytest.mark.parametrize("ntiles", [0, 1, 33, 384, 2048])
def test_chunk_split_with_tiles(hx, ntiles):
    """The split of a plan with tiles covers [0, n) once, in multiples of four histories and at
    most 8 blocks per SM."""
    hx.hx_chunk_split.restype = None
    blocks, per = ctypes.c_int(), ctypes.c_longlong()
    rng = np.random.default_rng(ntiles)
    ns = [1, 3, 4, 5, 255, 256, 257, 5064, 180000, 550000, 9000000, 1 << 25]
    for sm in (1, 7, 152):
        for n in ns + [int(x) for x in rng.integers(1, 1 << 25, 100)]:
            hx.hx_chunk_split(ctypes.c_longlong(n), sm, ntiles, ctypes.byref(blocks), ctypes.byref(per))
            b, p = blocks.value, per.value
            assert p % 4 == 0 and p > 0 and 1 <= b <= 8 * sm, (n, sm, b, p)
            assert b * p >= n and (b - 1) * p < n, (n, sm, b, p)
