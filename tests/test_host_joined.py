"""Event walks of all types in one joined tile (hd_geom.cuh), compiled for the
host, against the CPU oracle's voxel sets: the counts of many segments together,
on adversarial segments and generic ones, every update inside the tile, and as
many equal walks as a part can hold.  Runs without a GPU."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

from tests.test_host_events import _generic
from tests.test_oracle_pins import _random_segments

HERE = os.path.dirname(os.path.abspath(__file__))
SRC = os.path.join(HERE, "host_harness", "host_joined.cu")
I32P, U8P = ctypes.POINTER(ctypes.c_int32), ctypes.POINTER(ctypes.c_uint8)


@pytest.fixture(scope="module")
def hx(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    out = str(tmp_path_factory.mktemp("hx") / "libhostjoined.so")
    subprocess.check_call([nvcc, "-O2", "-std=c++17", "-Xcompiler", "-fPIC", "-shared",
                           "-gencode", "arch=compute_103a,code=sm_103a",
                           "-diag-suppress", "20014", "-o", out, SRC,
                           "-I", os.path.join(HERE, "..", "include")])
    return ctypes.CDLL(out)


def _joined(hx, segs, dims, direct):
    segs = np.ascontiguousarray(segs, np.int32)
    counts = np.zeros(int(np.prod(dims)), np.int32)
    skipped = np.zeros(len(segs), np.uint8)
    n = hx.hx_joined(segs.ctypes.data_as(I32P), len(segs), *dims, direct,
                     counts.ctypes.data_as(I32P), skipped.ctypes.data_as(U8P))
    assert n >= 0, n
    return counts, skipped, n


@pytest.mark.parametrize("dims,direct", [((5, 4, 1), 1), ((1, 1, 1), 1), ((1, 7, 1), 1),
                                         ((9, 1, 1), 1), ((40, 30, 1), 1), ((17, 64, 1), 1),
                                         ((4096, 2, 1), 1), ((2, 4000, 1), 1), ((237, 237, 1), 1),
                                         ((12, 11, 3), 0), ((40, 30, 2), 0)])
def test_joined_tiles_equal_oracle(oracle_mod, hx, dims, direct):
    rng = np.random.default_rng(sum(dims) + 11)
    segs = list(_random_segments(rng, 1000, dims)) + list(_generic(rng, 1500, dims))
    flat = np.array([np.concatenate([a, b]) for a, b in segs], np.int32)
    counts, skipped, n = _joined(hx, flat, dims, direct)
    want = np.zeros(int(np.prod(dims)), np.int64)
    for (a, b), skip in zip(segs, skipped):
        if not skip:
            want[oracle_mod.voxel_set(np.asarray(a, np.int32), np.asarray(b, np.int32), *dims)] += 1
    assert n > 200 and np.array_equal(counts, want)


@pytest.mark.parametrize("seg", [((-1.37, 3.31, 0.5), (41.23, 20.17, 0.5)), ((41.23, 3.31, 0.5), (-1.37, 20.17, 0.5)),
                                 ((3.31, -1.29, 0.5), (12.73, 31.19, 0.5)), ((12.73, -1.29, 0.5), (3.31, 31.19, 0.5)),
                                 ((0.23, 0.11, 0.5), (39.91, 0.37, 0.5)), ((39.61, 0.13, 0.5), (39.79, 29.93, 0.5))])
def test_most_walks_of_a_part(oracle_mod, hx, seg):
    """32736 equal walks: neither half of a word, nor a sum of them, overflows."""
    dims = (40, 30, 1)
    a, b = (np.round(65536 * np.array(p)).astype(np.int32) for p in seg)
    counts, skipped, n = _joined(hx, np.tile(np.concatenate([a, b]), (32736, 1)), dims, 1)
    want = np.zeros(1200, np.int64)
    want[oracle_mod.voxel_set(a, b, *dims)] = 32736
    assert n == 32736 and not skipped.any() and np.array_equal(counts, want)
