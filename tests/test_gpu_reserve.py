"""What hd_scan_reserve promises ends with the buffers it made: page-locked adds of as
many histories are read in place while it holds, and copied beside the traversal
again once a change of tuning has dropped the buffers."""
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


def test_reservation_and_tuning(hd):
    n, g = (3 << 20) + 1, synth.Geometry(24, 20, 12, 1.0, 1.0, 2.0, 30.0)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(n)
    u = torch.rand((6, n), generator=gen, device="cuda")
    u[0] *= 360.0
    u[1:5] = 24.0 * u[1:5] - 12.0
    u[5] *= 10.0
    host = torch.empty((6, n), pin_memory=True).copy_(u)

    def add(s, rows):
        """Kernels of an add, and its counts."""
        s.reset()
        before = s.profile()["kernel_launches"]
        s.add([rows[k] for k in range(6)])
        kernels = s.profile()["kernel_launches"] - before
        return kernels, s.counts(hd.HD_MSC), s.counts(hd.HD_SM)

    with hd.Scan(g) as s:
        one, N, M = add(s, u)
        s.reserve(n)
        got = [add(s, host)]
        s.reset()
        hd.hd_scan_set_tuning(s.handle, hd.hd_tuning(1024, 12, 30000, 0))
        got.append(add(s, host))
    assert got[0][0] == one and got[1][0] > one
    for _, x, y in got:
        assert np.array_equal(x, N) and np.array_equal(y, M)
