"""Regions grown along long rows (more words than a warp takes at a time) and in
slices of few rows in the hull diagnostics, against the oracle, bit for bit:
serpentine corridors, corridors from the sides alone, random masks, and weak edges
that run along the rows."""
import numpy as np
import pytest

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


def _slices(nx, ny):
    rng = np.random.default_rng(nx + ny)
    m = np.zeros((ny, nx), np.uint8)
    m[1::2] = 1
    m[1::2, 0] = m[1::2, -1] = 0
    for i, y in enumerate(range(1, ny - 2, 2)):
        m[y:y + 3, nx - 2 if i % 2 == 0 else 1] = 1
    m[ny // 2, :nx // 3] = 1
    side = np.zeros((ny, nx), np.uint8)
    side[1:-1] = 1
    side[ny // 2, nx // 2:nx // 2 + 3] = 0
    gaps = side.copy()
    gaps[:, 31::64] = rng.random((ny, gaps[:, 31::64].shape[1])) < 0.8
    return np.stack([m, m[:, ::-1], side, gaps, gaps[:, ::-1]] +
                    [(rng.random((ny, nx)) < d).astype(np.uint8) for d in (0.55, 0.7, 0.97)])


@pytest.mark.parametrize("nx,ny", [(640, 33), (641, 15), (672, 16), (673, 17), (1023, 3), (1025, 40),
                                   (2080, 7), (4100, 20), (33, 8), (700000, 1), (31, 5000)])
def test_fill(hd, oracle_mod, nx, ny):
    v = _slices(nx, ny) if nx * ny < 400000 else \
        (np.random.default_rng(1).random((2, ny, nx)) < 0.9).astype(np.uint8)
    dims = (nx, ny, len(v))
    got = hd.hd_fill_enclosed(torch.from_numpy(np.ascontiguousarray(v).ravel()).cuda(), dims)
    assert np.array_equal(got.cpu().numpy(), oracle_mod.fill_enclosed(v.ravel(), dims))


@pytest.mark.parametrize("nx,ny", [(700, 12), (700, 20), (2100, 16), (1500, 40), (40, 9)])
def test_weak_edges_along_rows(hd, oracle_mod, nx, ny):
    yy, xx = np.mgrid[0:ny, 0:nx]
    line = (yy >= ny // 2 + (xx // 90) % 3).astype(np.uint32)
    strong = np.where(xx < 20, 1000, 330).astype(np.uint32)
    M = np.stack([100 + strong * line, 100 + strong[:, ::-1] * line,
                  np.random.default_rng(nx).integers(0, 5000, (ny, nx))]).astype(np.uint32)
    dims = (nx, ny, 3)
    for q in (0, 60):
        mt, he, H3 = hd.hd_sm_canny(torch.from_numpy(M.ravel().view(np.int32)).cuda(), dims, q_pct=q)
        ref = oracle_mod.sm_canny(M, dims, q_pct=q)
        assert np.array_equal(mt.cpu().numpy().view(np.uint32), ref["Mt"])
        assert np.array_equal(he.cpu().numpy(), ref["has_edge"])
        assert np.array_equal(H3.cpu().numpy(), ref["H3"])
