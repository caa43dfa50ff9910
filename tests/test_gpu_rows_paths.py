"""System-matrix rows where their passes can go wrong: hulls that leave the emit
pass fewer threads or lie in global memory, cols at every offset from a 32-byte
boundary (rows leave as whole sectors), runs of more than 32 voxels, one-voxel
planes.  Every row against the oracle, in path order."""
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


@pytest.mark.parametrize("dims,n,offset", [((230, 229, 28), 3000, 3), ((256, 255, 26), 3000, 0),
                                           ((63, 64, 9), 5000, 1), ((1, 300, 2), 1500, 7),
                                           ((300, 1, 2), 1500, 5), ((40, 40, 5), 1, 2)])
def test_rows(hd, oracle_mod, dims, n, offset):
    g = synth.Geometry(*dims, 1.0, 1.0, 1.5, float(max(dims)))
    h = synth.tiny_random_case(np.random.default_rng(sum(dims)), n, g, span=1.1)
    # along the axes: runs over the whole grid
    h.angle_deg[: n // 4] = np.tile([0, 90, 180, 270], n)[: n // 4]
    h.u_out[: n // 8] = h.u_in[: n // 8]
    dev = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in h.arrays()]
    with hd.Scan(g) as s:
        s.add(dev)
        s.finalize()
        hull = s.mask(hd.HD_MSC)
        ref_ptr, ref_cols = oracle_mod.system_rows(g, h, hull, threads=8)
        row_ptr = torch.full((n + 1,), -1, dtype=torch.int64, device="cuda")
        room = torch.full((len(ref_cols) + offset + 9,), -7, dtype=torch.int32, device="cuda")
        cols = room[offset:offset + len(ref_cols)]
        total = hd.hd_scan_system_rows(s.handle, hd.HD_MSC, *dev[:5], row_ptr,
                                       cols if len(ref_cols) else None)
        torch.cuda.synchronize()
    assert total == len(ref_cols)
    assert np.array_equal(row_ptr.cpu().numpy(), ref_ptr)
    got = room.cpu().numpy()
    assert np.array_equal(got[offset:offset + total], ref_cols)
    # nothing outside the rows is written
    assert np.all(got[:offset] == -7) and np.all(got[offset + total:] == -7)
