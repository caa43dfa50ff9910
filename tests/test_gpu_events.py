"""The tiled traversal's event walks on the GPU against the oracle, bit for bit,
where they can go wrong: odd and one-voxel-wide planes, strips, deep slabs,
the smallest job size (a bucket cut into many parts), more buckets than a
block lists at a time, lattice ties (the warp-shared fallback), and dilated
scans of all of these that have whole-plane tiles."""
import numpy as np
import pytest

from paper_1402_1720_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - CPU container
    pytest.skip("needs a CUDA GPU", allow_module_level=True)


@pytest.fixture(scope="module")
def hd():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1402_1720_gb300 import hulld
    hulld.load()
    return hulld


G = synth.Geometry


def _histories(g, n, ties):
    if ties:
        from tests.test_gpu_parity import _lattice_histories
        return _lattice_histories(np.random.default_rng(g.nx + 7), g, n)
    return synth.tiny_random_case(np.random.default_rng(g.nx * 1000 + g.ny), n, g, span=1.1)


def _scan_counts(hd, g, h, k=0, tuning=None):
    dev = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in h.arrays()]
    with hd.Scan(g) as s:
        if tuning is not None:
            hd.hd_scan_set_tuning(s.handle, tuning)
        if k:
            s.set_thick(k)
        s.add(dev)
        s.finalize()
        return s.counts(hd.HD_MSC), s.counts(hd.HD_SM)


@pytest.mark.parametrize("g,n,ties,tuning", [
    (G(1, 1, 3, 1.0, 1.0, 1.0, 3.0), 500, False, None),
    (G(1, 37, 2, 1.0, 1.0, 1.0, 30.0), 2000, False, None),
    (G(53, 1, 4, 1.0, 2.0, 1.0, 40.0), 2000, True, None),
    (G(97, 64, 5, 1.0, 1.0, 2.0, 80.0), 20000, False, (1024, 12, 256, 0)),
    (G(64, 97, 6, 1.0, 1.0, 2.0, 80.0), 20000, True, (256, 1, 32767, 3)),
    (G(300, 260, 3, 0.5, 0.5, 2.0, 120.0), 4000, False, (512, 32, 5000, 0)),
    (G(12, 10, 1200, 1.0, 1.0, 0.5, 20.0), 6000, False, None),
])
def test_thin(hd, oracle_mod, g, n, ties, tuning):
    h = _histories(g, n, ties)
    ref = oracle_mod.run(g, h)
    N, M = _scan_counts(hd, g, h, tuning=None if tuning is None else hd.hd_tuning(*tuning))
    assert np.array_equal(N, ref["N"]) and np.array_equal(M, ref["M"])


@pytest.mark.parametrize("g,ties", [(G(17, 40, 3, 1.0, 1.0, 2.0, 40.0), True),
                                    (G(40, 31, 2, 1.0, 1.0, 2.0, 40.0), False),
                                    (G(1, 25, 2, 1.0, 1.0, 2.0, 30.0), True),
                                    (G(22, 2, 2, 1.0, 1.0, 2.0, 30.0), True)])
@pytest.mark.parametrize("k", [1, 2, 16])
def test_dilated(hd, oracle_mod, g, ties, k):
    h = _histories(g, 3000, ties)
    ref = oracle_mod.accumulate_thick(g, h, k)
    N, M = _scan_counts(hd, g, h, k)
    assert np.array_equal(N, ref["N"]) and np.array_equal(M, ref["M"])
