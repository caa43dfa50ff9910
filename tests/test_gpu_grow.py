"""Regions grown tile by tile (32 rows by one word of bits) in the hull
diagnostics, at the edges of tiles: serpentine corridors that cross every tile
many times, weak edges that run diagonally through tile corners, and compared
volumes that start at odd addresses; against the oracle, bit for bit."""
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


@pytest.mark.parametrize("nx,ny", [(31, 33), (32, 32), (33, 64), (65, 97), (130, 31), (3, 200)])
@pytest.mark.parametrize("gap", [2, 3])
def test_serpentine_corridors(hd, oracle_mod, nx, ny, gap):
    """The mask is a one-voxel corridor winding through the slice from its border; the rows
    beside it are walls, with enclosed voxels in every third wall."""
    m = np.zeros((ny, nx), np.uint8)
    m[1::gap] = 1
    m[1::gap, 0] = m[1::gap, -1] = 0
    for i, y in enumerate(range(1, ny - gap, gap)):
        m[y:y + gap + 1, nx - 2 if i % 2 == 0 else 1] = 1
    m[1, 0] = 1
    vols = np.stack([m, m[:, ::-1], m[::-1], 1 - m])
    got = hd.hd_fill_enclosed(torch.from_numpy(np.ascontiguousarray(vols).ravel()).cuda(), (nx, ny, 4))
    assert np.array_equal(got.cpu().numpy(), oracle_mod.fill_enclosed(vols.ravel(), (nx, ny, 4)))


@pytest.mark.parametrize("nx,ny", [(64, 64), (70, 101), (33, 130)])
@pytest.mark.parametrize("slope", [1.0, -1.0, 0.4])
def test_weak_edges_across_tiles(hd, oracle_mod, nx, ny, slope):
    """An edge strong at one end and weak along a slanted line through the slice."""
    yy, xx = np.mgrid[0:ny, 0:nx]
    side = (yy - ny / 2) - slope * (xx - nx / 2) > 0
    step = np.where(xx < nx // 6, 1000, 330)
    M = (100 + step * side).astype(np.uint32)[None]
    M = np.concatenate([M, np.ascontiguousarray(M[:, ::-1]), np.full_like(M, 9)])
    for q in (0, 37, 100):
        mt, he, H3 = hd.hd_sm_canny(torch.from_numpy(M.ravel().view(np.int32)).cuda(), (nx, ny, 3), q_pct=q)
        ref = oracle_mod.sm_canny(M, (nx, ny, 3), q_pct=q)
        assert np.array_equal(mt.cpu().numpy().view(np.uint32), ref["Mt"])
        assert np.array_equal(he.cpu().numpy(), ref["has_edge"])
        assert np.array_equal(H3.cpu().numpy(), ref["H3"])


@pytest.mark.parametrize("dims", [(64, 64, 3), (61, 67, 2), (128, 96, 2), (4096, 1, 1), (1, 4097, 1)])
@pytest.mark.parametrize("shift", [0, 1, 16])
def test_compare_addresses(hd, oracle_mod, dims, shift):
    V = int(np.prod(dims))
    rng = np.random.default_rng(V + shift)
    h = rng.integers(0, 256, V + 32).astype(np.uint8) * (rng.random(V + 32) < 0.4)
    o = rng.integers(0, 256, V + 32).astype(np.uint8) * (rng.random(V + 32) < 0.3)
    h, o = h.astype(np.uint8), o.astype(np.uint8)
    c = hd.hd_hull_compare(torch.from_numpy(h).cuda()[shift:shift + V],
                           torch.from_numpy(o).cuda()[:V], dims).cpu().numpy()
    ref = oracle_mod.hull_compare((h[shift:shift + V] != 0).astype(np.uint8),
                                  (o[:V] != 0).astype(np.uint8), dims)
    nz = dims[2]
    assert np.array_equal(c[:nz], ref["extra_per_slice"])
    assert np.array_equal(c[nz:2 * nz], ref["missing_per_slice"])
    assert (c[2 * nz], c[2 * nz + 1]) == (ref["extra"], ref["missing"])
