"""Cells joined in one tile on the GPU (all walk types, one flush) against the
oracle, bit for bit: launches of many buckets with few walks each, on whole planes,
strips and deep slabs, lattice ties, the smallest parts (a joined cell cut into
several), more parts than a block lists at a time, and several scans at once."""
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


def _histories(g, n, ties=False):
    if ties:
        from tests.test_gpu_parity import _lattice_histories
        return _lattice_histories(np.random.default_rng(g.nz), g, n)
    return synth.tiny_random_case(np.random.default_rng(g.nx + n), n, g, span=1.1)


@pytest.mark.parametrize("g,n,ties,tuning", [
    (G(40, 36, 80, 1.0, 1.0, 1.0, 40.0), 9000, False, None),
    (G(36, 40, 90, 1.0, 1.0, 1.0, 40.0), 9000, True, None),
    (G(300, 260, 60, 0.5, 0.5, 1.0, 120.0), 5000, False, None),
    (G(40, 36, 200, 1.0, 1.0, 0.5, 40.0), 9000, False, (512, 12, 32767, 3)),
    (G(33, 29, 50, 1.0, 1.0, 1.0, 40.0), 60000, False, (256, 4, 256, 0)),
    (G(9, 11, 1900, 1.0, 1.0, 0.25, 20.0), 4000, False, None),
    (G(1, 30, 60, 1.0, 1.0, 1.0, 30.0), 3000, True, None),
])
@pytest.mark.parametrize("chunks", [1, 3])
def test_scans(hd, oracle_mod, g, n, ties, tuning, chunks):
    h = _histories(g, n, ties)
    ref, dev = oracle_mod.run(g, h), _dev(h)
    edges = [n * k // chunks for k in range(chunks + 1)]
    with hd.Scan(g) as s:
        if tuning is not None:
            hd.hd_scan_set_tuning(s.handle, hd.hd_tuning(*tuning))
        for a, b in zip(edges, edges[1:]):
            s.add([c[a:b] for c in dev])
        s.finalize()
        assert np.array_equal(s.counts(hd.HD_MSC), ref["N"])
        assert np.array_equal(s.counts(hd.HD_SM), ref["M"])


@pytest.mark.parametrize("graph", [True, False])
def test_batch(hd, oracle_mod, graph):
    grids = [G(40, 36, 40, 1.0, 1.0, 1.0, 40.0), G(64, 20, 30, 1.0, 1.0, 1.0, 50.0),
             G(20, 24, 3, 1.0, 1.0, 2.0, 30.0), G(130, 90, 33, 0.5, 0.5, 1.0, 60.0)]
    hs = [_histories(g, n) for g, n in zip(grids, (3000, 500, 2000, 4000))]
    refs, st = [oracle_mod.run(g, h) for g, h in zip(grids, hs)], torch.cuda.Stream()
    scans, devs = [hd.Scan(g) for g in grids], [_dev(h) for h in hs]
    torch.cuda.synchronize()
    with hd.Batch() as b:
        b.set_graph(graph)
        for _ in range(2):
            for s, d in zip(scans, devs):
                b.add(s, d)
            b.run(hd.HD_BATCH_RESET | hd.HD_BATCH_FINALIZE, st)
            torch.cuda.synchronize()
            for s, r in zip(scans, refs):
                assert np.array_equal(s.counts(hd.HD_MSC), r["N"])
                assert np.array_equal(s.counts(hd.HD_SM), r["M"])
    for s in scans:
        s.close()
