"""A batch's captured graph is replayed only for the scans it holds: not after a
change of their tuning that keeps the block size, not for a new scan that has
taken a destroyed one's memory, not after their buffers have grown."""
import numpy as np
import pytest

from paper_1402_1720_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - CPU container
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

GRID = synth.Geometry(40, 36, 9, 1.0, 1.0, 2.0, 40.0)


@pytest.fixture(scope="module")
def hd():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1402_1720_gb300 import hulld
    hulld.load()
    return hulld


def _histories(n):
    h = synth.tiny_random_case(np.random.default_rng(n), n, GRID, span=1.1)
    return h, [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in h.arrays()]


def _run(hd, b, s, dev, st):
    """Whether the run captured a graph."""
    before = b.stats()["graph_captures"]
    b.add(s, dev)
    b.run(hd.HD_BATCH_RESET | hd.HD_BATCH_FINALIZE, st)
    torch.cuda.synchronize()
    return b.stats()["graph_captures"] > before


def _check(hd, s, ref):
    assert np.array_equal(s.counts(hd.HD_MSC), ref["N"])
    assert np.array_equal(s.counts(hd.HD_SM), ref["M"])
    assert np.array_equal(s.mask(hd.HD_MSC), ref["H2"])
    assert np.array_equal(s.mask(hd.HD_SM), ref["H3"])


@pytest.mark.parametrize("change", [dict(slab_depth=3), dict(job_size=256), dict(refill=3)])
def test_tuning_changed(hd, oracle_mod, change):
    h, dev = _histories(2000)
    ref, st = oracle_mod.run(GRID, h), torch.cuda.Stream()
    torch.cuda.synchronize()
    with hd.Batch() as b, hd.Scan(GRID) as s:
        assert _run(hd, b, s, dev, st)
        assert not _run(hd, b, s, dev, st)
        _check(hd, s, ref)
        for tuning in (change, {}):
            t = dict(threads=1024, refill=12, job_size=32767, slab_depth=0)
            t.update(tuning)
            s.reset()
            hd.hd_scan_set_tuning(s.handle, hd.hd_tuning(**t))
            assert _run(hd, b, s, dev, st)
            _check(hd, s, ref)


def test_scan_made_anew(hd, oracle_mod):
    h, dev = _histories(2000)
    st = torch.cuda.Stream()
    torch.cuda.synchronize()
    with hd.Batch() as b:
        for k, hit in enumerate((1.0, 5.0, 12.0, 1.0)):
            p = hd.hd_params_default()
            p.wepl_hit_gt = hit
            p.msc_nt = 2 + k
            with hd.Scan(GRID, p) as s:
                assert _run(hd, b, s, dev, st)
                assert not _run(hd, b, s, dev, st)
                _check(hd, s, oracle_mod.run(GRID, h, oracle_mod.Params(tau_h=hit, nt=2 + k)))


def test_buffers_grown(hd, oracle_mod):
    (h, dev), (big, bigdev) = _histories(500), _histories(30000)
    ref, st = oracle_mod.run(GRID, h), torch.cuda.Stream()
    with hd.Batch() as b, hd.Scan(GRID) as s:
        assert _run(hd, b, s, dev, st)
        s.reset()
        s.add(bigdev)
        s.finalize()
        torch.cuda.synchronize()
        _check(hd, s, oracle_mod.run(GRID, big))
        assert _run(hd, b, s, dev, st)
        _check(hd, s, ref)


@pytest.mark.parametrize("graph", [True, False])
@pytest.mark.parametrize("how", ["set_thick", "set_thick_distance"])
def test_thick_rays_set_after_queueing(hd, oracle_mod, how, graph):
    """Refused as at queueing; the scan and the batch work on."""
    h, dev = _histories(2000)
    ref, st = oracle_mod.run(GRID, h), torch.cuda.Stream()
    torch.cuda.synchronize()
    with hd.Batch() as b, hd.Scan(GRID) as s:
        b.set_graph(graph)
        for _ in range(2):
            b.add(s, dev)
            getattr(s, how)(2)
            with pytest.raises(hd.HDError) as e:
                b.run(hd.HD_BATCH_RESET | hd.HD_BATCH_FINALIZE, st)
            assert e.value.status == hd.HD_ERR_STATE
            getattr(s, how)(0)
            _run(hd, b, s, dev, st)
            _check(hd, s, ref)
            s.reset()
