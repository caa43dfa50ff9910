"""Page-locked histories that are copied in parts beside the traversal, against
the same histories on the device: evenly spaced columns and columns of their
own, several adds on one stream, dilated and Euclidean thick rays, and the
smallest count that is copied."""
import numpy as np
import pytest

from paper_1402_1720_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - CPU container
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

LEAST = 3 << 20


@pytest.fixture(scope="module")
def hd():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1402_1720_gb300 import hulld
    hulld.load()
    return hulld


def _rows(n):
    """6 x n columns of a small grid, made on the device and copied to page-locked memory."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(n)
    u = torch.rand((6, n), generator=gen, device="cuda")
    u[0] = torch.sort(360.0 * u[0]).values
    u[1:5] = 24.0 * u[1:5] - 12.0
    u[4] = u[2] + 0.1 * u[4]
    u[5] *= 40.0
    host = torch.empty((6, n), dtype=torch.float32, pin_memory=True)
    host.copy_(u)
    return u, host


def _counts(hd, s):
    torch.cuda.synchronize()
    return [s.counts(m) for m in (hd.HD_MSC, hd.HD_SM)] + [s.mask(hd.HD_SM)]


@pytest.mark.parametrize("n,how", [(LEAST, "thin"), (LEAST + 1, "thin"), (7_000_003, "thin"),
                                   (LEAST + 5, "thick"), (LEAST + 6, "distance")])
@pytest.mark.parametrize("columns", ["rows", "last apart", "all apart"])
def test_parts(hd, n, how, columns):
    g = synth.Geometry(24, 20, 12, 1.0, 1.0, 2.0, 30.0)
    dev, host = _rows(n)
    cols = [host[k] for k in range(6)]
    if columns == "last apart":
        cols[5] = torch.empty(n, dtype=torch.float32, pin_memory=True).copy_(host[5])
    if columns == "all apart":  # allocations of one size, which may lie evenly spaced
        cols = [torch.empty(n, dtype=torch.float32, pin_memory=True).copy_(c) for c in cols]
    with hd.Scan(g) as a, hd.Scan(g) as b:
        for s in (a, b):
            if how == "thick":
                s.set_thick(1)
            if how == "distance":
                s.set_thick_distance(1.2)
        st = torch.cuda.Stream()
        torch.cuda.synchronize()
        a.add([dev[k] for k in range(6)])
        a.add([dev[k][:1000] for k in range(6)])
        a.finalize()
        b.add(cols, st)
        b.add([c[:1000] for c in cols], st)
        b.finalize(st)
        for _ in range(2):
            for x, y in zip(_counts(hd, a), _counts(hd, b)):
                assert np.array_equal(x, y)
            if how == "distance":
                break
            a.add([dev[k] for k in range(6)])
            a.finalize()
            b.add(cols, st)  # the staging of the add before is used again
            b.finalize(st)


def test_reserved_adds_allocate_nothing(hd):
    """An add that was reserved for neither allocates nor changes its result."""
    g = synth.Geometry(24, 20, 12, 1.0, 1.0, 2.0, 30.0)
    n = LEAST + 7
    dev, host = _rows(n)
    with hd.Scan(g) as a, hd.Scan(g) as b:
        a.add([dev[k] for k in range(6)])
        a.finalize()
        b.reserve(n)
        b.add([dev[k][:8] for k in range(6)])
        b.reset()
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        b.add([host[k] for k in range(6)])
        b.finalize()
        torch.cuda.synchronize()
        assert torch.cuda.mem_get_info()[0] == free
        for x, y in zip(_counts(hd, a), _counts(hd, b)):
            assert np.array_equal(x, y)
