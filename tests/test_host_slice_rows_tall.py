"""The closed form of Euclidean rows on volumes much taller than wide, compiled for the
host: a path a little inclined keeps it (only the centres of its own slices have to
project onto the segment), its certain rows equal the exact search, and no row with
voxels is missed.  Runs without a GPU."""
import ctypes
import math

import numpy as np
import pytest

from tests.test_host_slice_rows import hx  # noqa: F401  (the compiled harness)


@pytest.mark.parametrize("dims,vox,T,tilt,d0", [((24, 24, 300), (1.0, 1.0, 4.0), 30.0, 3.0, 1.5),
                                                ((24, 24, 300), (1.0, 1.0, 4.0), 30.0, 20.0, 6.0),
                                                ((16, 20, 200), (1.0, 0.8, 0.5), 20.0, 4.0, 0.7)])
def test_inclined_paths_in_tall_volumes(hx, dims, vox, T, tilt, d0):  # noqa: F811
    rng = np.random.default_rng(dims[2])
    half, hz = math.hypot(dims[0] * vox[0], dims[1] * vox[1]) / 2, dims[2] * vox[2] / 2
    closed = rows = hit = 0
    for _ in range(150):
        phi = rng.uniform(0, 2 * math.pi)
        c, s = math.cos(phi), math.sin(phi)
        u0, v0 = rng.uniform(-half, half), rng.uniform(-hz, hz) * 1.05
        u1, v1 = u0 + rng.normal(0, 1.0), v0 + rng.normal(0, tilt)
        W = [-T * c - u0 * s, -T * s + u0 * c, v0, T * c - u1 * s, T * s + u1 * c, v1]
        W = (ctypes.c_longlong * 6)(*[int(round(x * 65536)) for x in W])
        opened, cl = ctypes.c_longlong(0), ctypes.c_int(0)
        n = hx.hx_slice_rows(W, *dims, *[ctypes.c_float(v) for v in vox], ctypes.c_float(T),
                             ctypes.c_float(d0), 0, max(dims), ctypes.byref(opened), ctypes.byref(cl))
        assert n >= 0, (n, list(W))
        closed += cl.value
        rows += n
        hit += 1
    assert rows > 500
    if tilt < 5.0:
        assert closed > 0.8 * hit, (closed, hit)
