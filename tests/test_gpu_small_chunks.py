"""A scan fed in chunks of very different sizes, against the oracle bit for bit:
one history, fewer than the ingest blocks, few buckets with whole blocks to
themselves, buckets that span several blocks, and full launches, one after
another on the same scratch."""
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


@pytest.mark.parametrize("thick", [0, 1])
@pytest.mark.parametrize("g,chunks", [
    (G(40, 36, 1, 1.0, 1.0, 2.0, 40.0), [1, 31, 700, 20_000, 5, 60_000, 2]),
    (G(33, 29, 40, 1.0, 1.0, 1.0, 40.0), [3000, 12, 50_000, 153, 3000]),
    (G(130, 72, 33, 0.9, 0.9, 1.5, 90.0), [5064, 1, 5064, 90_000, 40]),
])
def test_chunks(hd, oracle_mod, g, chunks, thick):
    h = synth.tiny_random_case(np.random.default_rng(g.nx + g.nz), sum(chunks), g, span=1.1)
    order = np.argsort(h.arrays()[0], kind="stable")  # by gantry angle, as they arrive
    h = h.take(order)
    ref = oracle_mod.accumulate_thick(g, h, thick) if thick else oracle_mod.run(g, h)
    dev = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in h.arrays()]
    edges = np.concatenate([[0], np.cumsum(chunks)])
    with hd.Scan(g) as s:
        if thick:
            s.set_thick(thick)
        for _ in range(2):
            s.reset()
            for a, b in zip(edges, edges[1:]):
                s.add([c[a:b] for c in dev])
            s.finalize()
            assert np.array_equal(s.counts(hd.HD_MSC), ref["N"])
            assert np.array_equal(s.counts(hd.HD_SM), ref["M"])
