"""thor_coarse_grain over maps with long member lists: refused maps do no work
that grows with a list, lists with a long segment are built in another way
than short ones and give the same sums in the same order."""

import time

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1607_05535_gb300 as thor
import workloads as wls
from paper_1607_05535_gb300 import closure as cl


def test_refused_maps_cost_no_more_than_their_count():
    """An all-zero map and one with an index out of range besides: every fine
    column of glevel 6 in one list. Ranking 40962 members against each other
    would be 5e7 dependent steps of one warp, a good part of a second; the
    count takes some 0.1 ms."""
    wl = wls.HS_G4.with_(nv=4)
    su = cl.make_setup(wl, 6, 2, thor.THOR_MIXED, None)
    try:
        before = thor.thor_state_get_all(su.coarse, su.ncol_c, su.nv)
        maps = [np.zeros(su.ncol_f, np.int32), np.zeros(su.ncol_f, np.int32)]
        maps[1][-1] = su.ncol_c
        thor.thor_coarse_grain(su.fine, su.scratch, su.fmap)      # the first call allocates the scratch
        for m in maps:
            with pytest.raises(thor.ThorError):
                thor.thor_coarse_grain(su.fine, su.coarse, m)
            t = time.perf_counter()
            with pytest.raises(thor.ThorError):
                thor.thor_coarse_grain(su.fine, su.coarse, m)
            assert time.perf_counter() - t < 0.02
        for a, b in zip(before, thor.thor_state_get_all(su.coarse, su.ncol_c, su.nv)):
            assert np.array_equal(a, b)
    finally:
        cl.destroy_setup(su)


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("longest", [512, 513, 1200])
def test_long_lists(longest, precision):
    """Coarse column 3 gets 'longest' members, at and above the length up to
    which lists are ranked on the device (512). Columns that keep their
    members keep their sums, bit for bit, whichever way the lists are built."""
    wl = wls.HS_G4.with_(nv=5)
    su = cl.make_setup(wl, 5, 2, thor.THOR_FP64 if precision == "fp64" else thor.THOR_MIXED, None)
    try:
        nv, ncf, ncc = su.nv, su.ncol_f, su.ncol_c
        if precision == "mixed":
            thor.thor_tune(su.fine, thor.THOR_TUNE_COMPENSATED, 0)
        thor.thor_step(su.fine, 1, wl.n_small, wl.dt)
        rng = np.random.default_rng(5)
        m = np.full(ncf, -1, np.int32)
        order = rng.permutation(ncf)
        m[order[:longest]] = 3
        rest = order[longest:]
        cols = np.array([c for c in range(ncc) if c != 3], np.int32)
        m[rest] = np.concatenate([cols, rng.choice(cols, rest.size - cols.size)])
        assert np.bincount(m, minlength=ncc).max() == longest
        thor.thor_coarse_grain(su.fine, su.coarse, m)
        # the same members outside of column 3, whose own go to columns 0 to 2 in short lists besides one
        short = m.copy()
        moved = np.flatnonzero(m == 3)[1:]
        short[moved] = np.arange(moved.size) % 3
        thor.thor_coarse_grain(su.fine, su.scratch, short)
        same = np.arange(ncc) > 3
        area = thor.thor_grid_areas(su.fine_grid)
        w = np.zeros(ncc)
        np.add.at(w, m, area)
        for f in (thor.THOR_FIELD_W, thor.THOR_FIELD_RHOTHETA, thor.THOR_FIELD_MOM):
            a, b = (thor.thor_state_get(s, f, ncc, nv) for s in (su.coarse, su.scratch))
            assert np.array_equal(a[same], b[same])
        fine = thor.thor_state_get(su.fine, thor.THOR_FIELD_W, ncf, nv)
        want = np.zeros((ncc, nv + 1))
        np.add.at(want, m, fine * (area / w[m])[:, None])
        want[:, 0] = want[:, nv] = 0.0
        # one rounding to the storage type, n float64 additions on both sides
        eps = (2.0 ** -24 if precision == "mixed" else 0.0) + 4 * ncf * 2.0 ** -53
        got = thor.thor_state_get(su.coarse, thor.THOR_FIELD_W, ncc, nv)
        assert np.max(np.abs(got - want)) <= eps * np.max(np.abs(fine))
        again = thor.thor_state_get_all(su.coarse, ncc, nv)
        thor.thor_coarse_grain(su.fine, su.coarse, m)
        for a, b in zip(again, thor.thor_state_get_all(su.coarse, ncc, nv)):
            assert np.array_equal(a, b)
    finally:
        cl.destroy_setup(su)
