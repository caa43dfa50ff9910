"""Batches by every route, against the oracle bit for bit: one scan or many,
several rounds of the same scans, paths that leave the tiled pass (all scans'
in one launch), and a captured graph before and after a direct run that used
the batch's tables for other scans."""
import numpy as np
import pytest

from paper_1402_1720_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - CPU container
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

G = synth.Geometry
GRIDS = [G(33, 29, 40, 1.0, 1.0, 0.5, 40.0), G(20, 24, 3, 1.0, 1.0, 2.0, 30.0),
         G(64, 50, 7, 1.0, 1.0, 2.0, 50.0)]


@pytest.fixture(scope="module")
def hd():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1402_1720_gb300 import hulld
    hulld.load()
    return hulld


def _histories(k, n):
    """A third of the paths are steep: in a small chunk they exceed the pair budget."""
    g = GRIDS[k]
    h = synth.tiny_random_case(np.random.default_rng(10 * k + n), n, g, span=1.1)
    cols = [np.array(a) for a in h.arrays()]
    top = 0.45 * g.nz * g.sz
    cols[2][::3], cols[4][::3] = -top, top
    return synth.Histories(*cols)


def _dev(h):
    return [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in h.arrays()]


def _check(hd, s, ref):
    torch.cuda.synchronize()
    assert np.array_equal(s.counts(hd.HD_MSC), ref["N"])
    assert np.array_equal(s.counts(hd.HD_SM), ref["M"])
    assert np.array_equal(s.mask(hd.HD_SM), ref["H3"])


@pytest.mark.parametrize("graph", [True, False])
@pytest.mark.parametrize("sizes", [[40], [3000, 1, 20], [5, 700, 60]])
def test_scans_and_rounds(hd, oracle_mod, sizes, graph):
    hs = [_histories(k, n) for k, n in enumerate(sizes)]
    refs = [oracle_mod.run(GRIDS[k], h) for k, h in enumerate(hs)]
    twice = [oracle_mod.run(GRIDS[k], synth.Histories.concat([h, h])) for k, h in enumerate(hs)]
    devs, st = [_dev(h) for h in hs], torch.cuda.Stream()
    scans = [hd.Scan(GRIDS[k]) for k in range(len(sizes))]
    torch.cuda.synchronize()
    with hd.Batch() as b:
        b.set_graph(graph)
        for rounds, want in ((1, refs), (2, twice), (1, refs), (1, refs)):
            for _ in range(rounds):
                for s, d in zip(scans, devs):
                    b.add(s, d)
            b.run(hd.HD_BATCH_RESET | hd.HD_BATCH_FINALIZE, st)
            for s, r in zip(scans, want):
                _check(hd, s, r)
    for s in scans:
        s.close()


def test_graph_after_a_direct_run(hd, oracle_mod):
    """A captured run, then a direct one of other scans, then the captured one again."""
    hs = [_histories(k, 500) for k in range(3)]
    refs = [oracle_mod.run(GRIDS[k], h) for k, h in enumerate(hs)]
    devs, st = [_dev(h) for h in hs], torch.cuda.Stream()
    scans = [hd.Scan(GRIDS[k]) for k in range(3)]
    torch.cuda.synchronize()
    flags = hd.HD_BATCH_RESET | hd.HD_BATCH_FINALIZE
    with hd.Batch() as b:
        for group, stream in (((0, 1), st), ((2,), 0), ((0, 1), st)):
            for k in group:
                b.add(scans[k], devs[k])
            b.run(flags, stream)
            for k in group:
                _check(hd, scans[k], refs[k])
    for s in scans:
        s.close()
