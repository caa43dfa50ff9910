"""Masks and counts copied to the device at any alignment, against the host
copies; the bytes beside them stay as they were."""
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


@pytest.mark.parametrize("dims", [(1, 1, 1), (3, 5, 1), (16, 16, 4), (33, 29, 5), (200, 180, 32)])
@pytest.mark.parametrize("shift", [0, 1, 4, 16])
def test_alignments(hd, dims, shift):
    g = synth.Geometry(*dims, 1.0, 1.0, 1.0, 200.0)
    V = int(np.prod(dims))
    h = synth.tiny_random_case(np.random.default_rng(V), 3000, g, span=1.1)
    with hd.Scan(g) as s:
        s.add([torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in h.arrays()])
        s.finalize()
        for m in (hd.HD_SC, hd.HD_MSC, hd.HD_SM):
            buf = torch.full((V + 40,), 77, dtype=torch.uint8, device="cuda")
            s.mask(m, out=buf[shift:shift + V])
            got = buf.cpu().numpy()
            assert np.array_equal(got[shift:shift + V], s.mask(m))
            assert (got[:shift] == 77).all() and (got[shift + V:] == 77).all()
        for m in (hd.HD_MSC, hd.HD_SM):
            buf = torch.full((V + 40,), 77, dtype=torch.int32, device="cuda")
            s.counts(m, out=buf[shift:shift + V])
            got = buf.cpu().numpy()
            assert np.array_equal(got[shift:shift + V].view(np.uint32), s.counts(m))
            assert (got[:shift] == 77).all() and (got[shift + V:] == 77).all()
