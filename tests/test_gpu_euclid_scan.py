"""Scans set to a Euclidean distance on the GPU (the tiled path and what it hands
on) against the oracle, bit for bit: strips along y, rows of both axes and long
ones, anisotropic and extreme voxels, records without the closed form (trackers
inside the grid, axis-parallel paths), so few histories that no list of open rows
has room, and a scan in several chunks because its buffers were made for thin
paths."""
import numpy as np
import pytest

from paper_1402_1720_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - CPU container
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

G = synth.Geometry


@pytest.fixture(scope="module")
def hd():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1402_1720_gb300 import hulld
    hulld.load()
    return hulld


def _dev(h):
    return [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in h.arrays()]


def _scattered(g, n, sigma=0.02):
    """Paths through the grid at every angle, as an acquisition has them: a little off straight."""
    rng = np.random.default_rng(n + g.nx)
    half, hz = np.hypot(g.nx * g.sx, g.ny * g.sy) / 2, g.nz * g.sz / 2
    u, v = rng.uniform(-half, half, n), rng.uniform(-1.1 * hz, 1.1 * hz, n)
    cols = [rng.uniform(0, 360, n), u, v, u + rng.normal(0, sigma * half, n),
            v + rng.normal(0, 0.1 * hz, n), rng.choice([0.5, 3.0, 7.0], n)]
    return synth.Histories(*[np.ascontiguousarray(c, np.float32) for c in cols])


def _check(hd, s, ref):
    torch.cuda.synchronize()
    assert ref["N"].sum() + ref["M"].sum() > 0
    assert np.array_equal(s.counts(hd.HD_MSC), ref["N"])
    assert np.array_equal(s.counts(hd.HD_SM), ref["M"])


@pytest.mark.parametrize("g,n,d0", [
    (G(300, 260, 4, 0.7, 0.7, 2.0, 160.0), 1200, 2.3),      # two strips
    (G(60, 2000, 3, 1.0, 0.1, 2.0, 120.0), 600, 1.1),       # three, rows along y
    (G(4096, 150, 2, 0.05, 0.5, 2.0, 130.0), 200, 0.6),     # thirteen, rows of 4096
    (G(4096, 250, 1, 0.05, 0.5, 2.0, 140.0), 100, 0.6),     # more strips than the path takes
    (G(64, 48, 12, 1.0, 1.3, 0.8, 60.0), 2000, 2.5),
    (G(23, 17, 9, 1.0, 1.0, 2.5, 40.0), 2000, 0.3),
    (G(24, 24, 24, 1 / 64, 1 / 64, 1 / 64, 1.0), 1500, 0.02),
    (G(12, 10, 6, 64.0, 64.0, 64.0, 4000.0), 1500, 63.9),
    (G(40, 30, 6, 1.0, 1.0, 1.0, 12.0), 1500, 1.0),         # trackers inside the grid
    (G(24, 28, 300, 1.0, 1.0, 4.0, 40.0), 1500, 1.5),       # tall: far slices beyond the ends
])
@pytest.mark.parametrize("few", [False, True])
def test_scattered_paths(hd, oracle_mod, g, n, d0, few):
    h = _scattered(g, min(n, 40) if few else n)
    ref, dev = oracle_mod.accumulate_euclid(g, h, d0, threads=16), _dev(h)
    with hd.Scan(g) as s:
        s.set_thick_distance(d0)
        for _ in range(2):
            s.reset()
            s.add(dev)
            s.finalize()
            _check(hd, s, ref)


@pytest.mark.parametrize("g,d0", [(G(23, 17, 9, 1.0, 1.0, 2.5, 40.0), 1.7),
                                  (G(16, 40, 12, 0.5, 1.25, 0.75, 40.0), 0.9),
                                  (G(300, 250, 2, 0.2, 0.2, 3.0, 60.0), 1.0),
                                  (G(20, 7, 9, 2.0, 0.125, 0.0625, 100.0), 0.3)])
def test_paths_without_the_closed_form(hd, oracle_mod, g, d0):
    """Every direction, some rejected, some parallel to an axis or to the slices."""
    h = synth.tiny_random_case(np.random.default_rng(g.nx), 1500, g, span=1.3)
    h.u_out[:200] = h.u_in[:200]
    h.angle_deg[:200] = np.float32([0, 90, 180, 270] * 50)
    h.v_out[100:300] = h.v_in[100:300]
    h.u_in[400:410] = np.float32(5000.0)
    h.angle_deg[410:420] = np.float32(np.nan)
    ref, dev = oracle_mod.accumulate_euclid(g, h, d0, threads=16), _dev(h)
    with hd.Scan(g) as s:
        s.set_thick_distance(d0)
        s.add([c[:7] for c in dev])
        s.add([c[7:] for c in dev])
        s.finalize()
        _check(hd, s, ref)


def test_several_chunks(hd, oracle_mod):
    """Buffers made by thin adds hold fewer pairs than the thick rays of as many histories."""
    g, d0 = G(48, 40, 30, 1.0, 1.0, 1.0, 60.0), 4.0
    h = _scattered(g, 4000)
    ref, dev = oracle_mod.accumulate_euclid(g, h, d0, threads=16), _dev(h)
    thin = oracle_mod.run(g, h)
    with hd.Scan(g) as s:
        s.add(dev)
        s.finalize()
        _check(hd, s, thin)
        s.reset()
        s.set_thick_distance(d0)
        s.add(dev)
        s.finalize()
        _check(hd, s, ref)
        s.reset()
        s.set_thick_distance(0.0)
        s.add(dev)
        s.finalize()
        _check(hd, s, thin)
