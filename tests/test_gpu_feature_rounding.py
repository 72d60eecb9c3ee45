"""The neighbour anomalies of the closure's features in float states: the mean
over the neighbours minus the value, rounded to float32 once. With zero mean
and unit scale the feature is that number itself: at most half a unit in its
last place from the exact value of the stored floats, and 2^-44 of the
largest difference that enters it (the pairs' own rounding)."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1607_05535_gb300 as thor
import workloads as wls
from test_gpu_closure_tiles import _pair, _planes


@pytest.mark.parametrize("glevel, nv", [(2, 12), (3, 33)])
def test_anomalies_are_rounded_once(glevel, nv):
    p, wl = _pair(nv, thor.THOR_MIXED, glevel)
    try:
        thor.thor_step(p.state, 2, wl.n_small, 300.0)
        x = torch.empty((wl.ncol, 10 * nv), dtype=torch.float32, device="cuda")
        z = torch.zeros(10 * nv, device="cuda")
        thor.thor_closure_features(p.state, z, z + 1.0, x)
        torch.cuda.synchronize()
        f = _planes(p.state, nv, thor.THOR_MIXED)[:, :, :wl.ncol].astype(np.longdouble)
        nbr = thor.thor_grid_neighbours(p.grid)
        ok = nbr >= 0
        d = np.where(ok, f[:, :, np.where(ok, nbr, 0)] - f[..., None], 0.0)
        exact = (d.sum(-1) / ok.sum(1)).transpose(2, 0, 1).reshape(wl.ncol, -1)
        size = np.abs(d).max(-1).transpose(2, 0, 1).reshape(wl.ncol, -1)
        ulp = np.spacing(np.abs(exact).astype(np.float32)).astype(np.longdouble)
        err = np.abs(x.cpu().numpy()[:, 5 * nv:] - exact)
        assert (size > 0).mean() > 0.9
        assert (err <= (0.5 + 2.0 ** -16) * ulp + 2.0 ** -44 * size).all(), float((err / ulp).max())
    finally:
        p.close()
