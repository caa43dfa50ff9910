"""The passes of binned SC that keep an angle's bins in shared memory, against
the oracle: angles in and out of order, bins fuller than a table word holds,
bins in several windows, histories cut against other histories' statistics,
and vertical bins with many slices, one or none."""
import dataclasses

import numpy as np
import pytest
import torch

from paper_1402_1720_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hd():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1402_1720_gb300 import hulld
    hulld.load()
    return hulld


def _histories(rng, n, bp, angles, wide, ordered):
    """n histories over the bins' face; wide: slopes and WEPL over their whole range."""
    ang = rng.choice(np.asarray(angles, np.float64), n)
    if ordered:
        ang = np.sort(ang)
    um = rng.uniform(bp.u_lo_mm - 0.5, bp.u_lo_mm + bp.n_u * bp.u_bin_mm + 0.5, n)
    vm = rng.uniform(bp.v_lo_mm - 0.5, bp.v_lo_mm + bp.v_bins * bp.v_bin_mm + 0.5, n)
    s = 300.0 if wide else 1.5
    du, dv = rng.normal(0, s, n), rng.normal(0, s, n)
    wepl = np.where(rng.random(n) < 0.6, rng.normal(0.5, 0.3, n),
                    rng.uniform(-1024.0, 1024.0, n) if wide else rng.uniform(0, 150.0, n))
    cols = [ang, um - du / 2, vm - dv / 2, um + du / 2, vm + dv / 2, wepl]
    cols[0][rng.random(n) < 0.001] = np.nan
    cols[5][rng.random(n) < 0.001] = np.inf
    return synth.Histories(*[np.ascontiguousarray(c, np.float32) for c in cols])


def _check(hd, om, g, bp, h):
    dev = [torch.from_numpy(np.ascontiguousarray(a, np.float32)).cuda() for a in h.arrays()]
    ref = om.sc_binned(g, h, bp)
    with hd.Binned(g, bp) as b:
        b.run(dev)
        assert np.array_equal(b.bins(), ref["bins"])
        assert np.array_equal(b.image(hd.HD_BINNED_CARVED), ref["carved"])
        assert np.array_equal(b.image(hd.HD_BINNED_HULL), ref["mask"])
        st, rs = b.stats(), ref["stats"]
        for k, r in (("histories_binned", "binned"), ("histories_cut", "cut"),
                     ("bins_used", "bins_used"), ("bins_missed", "bins_missed"),
                     ("lines", "lines"), ("lines_outside", "lines_outside")):
            assert st[k] == rs[r], k
    return ref


@pytest.mark.parametrize("ordered", [True, False])
@pytest.mark.parametrize("wide", [False, True])
def test_angles_in_and_out_of_order(hd, oracle_mod, ordered, wide):
    """Negative angles, angles past 360 and on bin edges; every third of the bins' histories
    lies outside the face or is not binned."""
    g = synth.Geometry(24, 20, 7, 1.0, 1.0, 1.0, 40.0)
    bp = oracle_mod.BinnedParams(u_lo_mm=-6.0, n_u=12, v_lo_mm=-2.0, v_bin_mm=1.5, v_bins=3)
    h = _histories(np.random.default_rng(3), 60_000, bp, [-4.0, 2.0, 6.0, 358.0, 362.0, 719.0, 90.3],
                   wide, ordered)
    ref = _check(hd, oracle_mod, g, bp, h)
    assert ref["stats"]["cut"] > 0 or wide


@pytest.mark.parametrize("n", [18 * 152, 50_000, 400_000])
def test_bins_fuller_than_a_table_word(hd, oracle_mod, n):
    """Nine bins, one of them taking most histories at the ends of the value range."""
    g = synth.Geometry(16, 16, 4, 1.0, 1.0, 2.5, 30.0)
    bp = oracle_mod.BinnedParams(u_lo_mm=-1.5, n_u=3, v_lo_mm=-3.0, v_bin_mm=2.0, v_bins=3,
                                 k_sigma=1)
    rng = np.random.default_rng(n)
    h = _histories(rng, n, bp, [8.0], True, True)
    hot = rng.random(n) < 0.9
    sign = rng.choice([-1.0, 1.0], n, p=[0.02, 0.98]).astype(np.float32)
    cols = [np.array(a) for a in h.arrays()]
    for k, v in ((1, 511.9), (2, 511.9), (3, -511.9), (4, -511.9)):
        cols[k][hot] = (v * sign)[hot]
    cols[5][hot] = (1023.999 * sign)[hot]
    _check(hd, oracle_mod, g, bp, synth.Histories(*cols))


def test_windows_of_vertical_bins(hd, oracle_mod):
    """2000 x 5 bins of an angle: two rows of the statistics fit in shared memory."""
    g = synth.Geometry(64, 64, 6, 1.0, 1.0, 1.0, 60.0)
    bp = oracle_mod.BinnedParams(u_lo_mm=-62.5, u_bin_mm=0.0625, n_u=2000, v_lo_mm=-2.5,
                                 v_bin_mm=1.0, v_bins=5)
    h = _histories(np.random.default_rng(5), 2_000_000, bp, np.arange(10) * 36.0, False, True)
    _check(hd, oracle_mod, g, bp, h)


def test_cut_against_other_histories(hd, oracle_mod):
    """The cut pass judges histories that did not enter the statistics as one history at a time
    does: the kept sums of both routes agree, bins without statistics included."""
    g = synth.Geometry(24, 20, 7, 1.0, 1.0, 1.0, 40.0)
    bp = oracle_mod.BinnedParams(u_lo_mm=-6.0, n_u=12, v_lo_mm=-2.0, v_bin_mm=1.5, v_bins=3)
    rng = np.random.default_rng(6)
    dev = [[torch.from_numpy(np.array(a)).cuda() for a in
            _histories(rng, n, bp, angles, False, True).arrays()]
           for n, angles in ((40_000, [0.0, 4.0, 8.0]), (60_000, [4.0, 8.0, 12.0, 16.0]))]
    with hd.Binned(g, bp) as a, hd.Binned(g, bp) as b:
        for x in (a, b):
            x.add(dev[0])
        a.cut(dev[1])
        for k in range(0, 60_000, 1000):  # too few for a table
            b.cut([c[k:k + 1000] for c in dev[1]])
        a.finalize(), b.finalize()
        assert np.array_equal(a.bins(), b.bins())
        assert a.stats() == b.stats()
        assert a.bins()[:, 7].sum() > 0


@pytest.mark.parametrize("v_lo, v_bin, v_bins", [(-10.0, 20.0, 1), (-30.0, 4.0, 15), (1.3, 0.7, 9),
                                                 (-40.0, 0.0625, 600)])
def test_slices_per_vertical_bin(hd, oracle_mod, v_lo, v_bin, v_bins):
    """A bin over every slice, bins with two and three slices, one or none, slices without a
    bin, and more empty bins than slices."""
    g = synth.Geometry(33, 31, 11, 0.9, 1.1, 1.5, 40.0)
    bp = dataclasses.replace(oracle_mod.binned_params_for(g), v_lo_mm=v_lo, v_bin_mm=v_bin,
                             v_bins=v_bins)
    h = _histories(np.random.default_rng(7), 30_000, bp, np.arange(90) * 4.0, False, True)
    ref = _check(hd, oracle_mod, g, bp, h)
    assert ref["stats"]["lines"] > 0
