"""Dilated paths that do not fit the pair budget of a small chunk take the
global path: their dilation is the scan's there too."""
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


@pytest.mark.parametrize("k", [1, 3])
@pytest.mark.parametrize("n", [1, 2, 40])
def test_steep_paths(hd, oracle_mod, n, k):
    """Each path crosses nearly all of the 40 slices, more than a history's share of pairs."""
    g = synth.Geometry(41, 36, 40, 1.0, 1.0, 0.5, 40.0)
    rng = np.random.default_rng(n)
    u, d = rng.uniform(-12, 12, n), rng.choice([-1.0, 1.0], n)
    cols = [rng.uniform(0, 360, n), u, -18.0 * d, u + rng.normal(0, 1, n), 18.0 * d,
            rng.choice([0.0, 50.0], n)]
    h = synth.Histories(*[np.ascontiguousarray(c, np.float32) for c in cols])
    ref = oracle_mod.accumulate_thick(g, h, k)
    with hd.Scan(g) as s:
        s.set_thick(k)
        s.add([torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in h.arrays()])
        s.finalize()
        assert np.array_equal(s.counts(hd.HD_MSC), ref["N"])
        assert np.array_equal(s.counts(hd.HD_SM), ref["M"])
