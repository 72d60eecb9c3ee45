"""thor_coarse_grain over maps whose members are scattered, uneven or many per
coarse column (member lists longer than a warp), and the maps it refuses: an
index out of range, a coarse column without members. The reference sums run
over rising fine columns on the host in float64, as the kernel's do."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1607_05535_gb300 as thor
import workloads as wls
from paper_1607_05535_gb300 import closure as cl


def _map(kind, nf, nc, near):
    rng = np.random.default_rng(7)
    if kind == "near":
        return near
    m = rng.integers(0, nc, nf).astype(np.int32)
    m[rng.permutation(nf)[:nc]] = np.arange(nc)              # every coarse column has a member
    if kind == "one_large":                                  # most fine columns in one coarse column
        m[:] = 3
        m[rng.permutation(nf)[:nc]] = np.arange(nc)
    return m


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("gf,gc,kind", [(4, 3, "scattered"), (3, 1, "scattered"), (3, 2, "one_large"), (3, 0, "near")])
def test_member_lists(gf, gc, kind, precision):
    wl = wls.HS_G4
    su = cl.make_setup(wl, gf, gc, thor.THOR_FP64 if precision == "fp64" else thor.THOR_MIXED, None)
    nv, ncf, ncc = su.nv, su.ncol_f, su.ncol_c
    if precision == "mixed":
        thor.thor_tune(su.fine, thor.THOR_TUNE_COMPENSATED, 0)
    thor.thor_step(su.fine, 1, wl.n_small, wl.dt)
    fmap = _map(kind, ncf, ncc, su.fmap)
    thor.thor_coarse_grain(su.fine, su.coarse, fmap)
    area = thor.thor_grid_areas(su.fine_grid)
    w = np.zeros(ncc)
    np.add.at(w, fmap, area)
    got = thor.thor_state_get(su.coarse, thor.THOR_FIELD_W, ncc, nv)
    want = np.zeros((ncc, nv + 1))
    np.add.at(want, fmap, thor.thor_state_get(su.fine, thor.THOR_FIELD_W, ncf, nv) * (area / w[fmap])[:, None])
    want[:, 0] = want[:, nv] = 0.0
    # one rounding to the storage type; on both sides n float64 additions and the weights, n up to ncf
    eps = (2.0 ** -24 if precision == "mixed" else 0.0) + 4 * ncf * 2.0 ** -53
    scale = np.max(np.abs(thor.thor_state_get(su.fine, thor.THOR_FIELD_W, ncf, nv)))
    assert np.max(np.abs(got - want)) <= eps * scale
    again = thor.thor_state_get_all(su.coarse, ncc, nv)
    for bad in ("range", "negative", "empty"):
        m = fmap.copy()
        if bad == "empty":
            m[m == 1] = 0
        else:
            m[0] = ncc if bad == "range" else -1
        with pytest.raises(Exception):
            thor.thor_coarse_grain(su.fine, su.coarse, m)
        for a, b in zip(again, thor.thor_state_get_all(su.coarse, ncc, nv)):
            assert np.array_equal(a, b)                      # a refused map leaves the coarse state as it was
    # the same map again: the same sums, whatever the order of the lists
    thor.thor_coarse_grain(su.fine, su.coarse, fmap)
    for a, b in zip(again, thor.thor_state_get_all(su.coarse, ncc, nv)):
        assert np.array_equal(a, b)
