"""System rows of more histories than a chunk of path walks holds, against the
rows of the same histories in two calls."""
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


@pytest.mark.parametrize("n", [(1 << 22) + 1, (1 << 22) + 100_003])
def test_chunks(hd, n):
    g = synth.Geometry(16, 14, 4, 1.0, 1.0, 2.0, 20.0)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(n)
    u = torch.rand((6, n), generator=gen, device="cuda")
    u[0] *= 360.0
    u[1:5] = 24.0 * u[1:5] - 12.0
    u[5] *= 10.0
    with hd.Scan(g) as s:
        s.add([c[:3000].contiguous() for c in u])
        s.finalize()
        parts, cut = [], n // 2 + 1
        for a, b in ((0, n), (0, cut), (cut, n)):
            ptr = torch.empty(b - a + 1, dtype=torch.int64, device="cuda")
            cols = torch.empty((b - a) * 34, dtype=torch.int32, device="cuda")
            total = hd.hd_scan_system_rows(s.handle, hd.HD_SC, *[u[k, a:b] for k in range(5)], ptr, cols)
            parts.append((ptr, cols[:total]))
        torch.cuda.synchronize()
    (ptr, cols), (p0, c0), (p1, c1) = parts
    assert len(cols) > 1_000_000
    assert torch.equal(cols, torch.cat([c0, c1]))
    assert torch.equal(ptr, torch.cat([p0, p1[1:] + p0[-1]]))
