"""The closure's correction itself: a state stepped with it minus the same state
stepped without is dt (y out_std + out_mean), the momentum projected onto the
tangent plane, with y the network's output on the state's features. Level
counts that fill the 32 x 32 tiles and that do not; whole-grid pass and batched pass."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1607_05535_gb300 as thor
from test_gpu_closure_tiles import _pair, _planes


@pytest.mark.parametrize("tc", [1, 2])
@pytest.mark.parametrize("precision", [thor.THOR_FP64, thor.THOR_MIXED])
@pytest.mark.parametrize("nv", [5, 32, 33])
def test_increment(nv, precision, tc):
    dt = 300.0
    p, wl = _pair(nv, precision)
    q, _ = _pair(nv, precision)
    n = wl.ncol
    net = thor.thor_mlp_create([10 * nv, 24, 40, 5 * nv], 50 if tc == 2 else n, seed=3)
    try:
        thor.thor_mlp_tune(net, thor.THOR_MLP_TUNE_TCGEN05, tc)
        dev = lambda a: torch.tensor(np.asarray(a, np.float32), device="cuda")
        raw = torch.empty((n, 10 * nv), device="cuda")
        thor.thor_closure_features(p.state, dev(np.zeros(10 * nv)), dev(np.ones(10 * nv)), raw)
        torch.cuda.synchronize()
        mean, std = raw.mean(0), raw.std(0) + 1e-6
        # corrections of about a hundredth of each field
        size = np.abs(_planes(p.state, nv, precision)[:, :, :n]).max(axis=(1, 2)).astype(np.float64) + 1e-6
        ostd = np.repeat(0.01 / dt * size, nv).astype(np.float32)
        omean = (0.3 * ostd * np.linspace(-1.0, 1.0, 5 * nv)).astype(np.float32)
        x = torch.empty((n, 10 * nv), device="cuda")
        thor.thor_closure_features(p.state, mean, std, x)
        y = torch.empty((n, 5 * nv), device="cuda")
        torch.cuda.synchronize()
        for c in range(0, n, 50 if tc == 2 else n):
            e = min(n, c + (50 if tc == 2 else n))
            xb, yb = x[c:e].contiguous(), torch.empty((e - c, 5 * nv), device="cuda")
            thor.thor_mlp_forward(net, xb, yb)
            y[c:e] = yb
        torch.cuda.synchronize()
        scale = [dev(ostd), dev(omean)]                           # the closure reads them until it is detached
        torch.cuda.synchronize()
        thor.thor_closure_attach(p.state, net, mean, std, scale[1], scale[0], period=1)
        for s in (p.state, q.state):
            thor.thor_step(s, 1, wl.n_small, dt)
        a, b = (_planes(s, nv, precision)[:, :, :n].astype(np.float64) for s in (p.state, q.state))
        thor.thor_closure_attach(p.state, None)
        tau = (y.cpu().numpy().astype(np.float64) * ostd + omean).reshape(n, 5, nv).transpose(1, 2, 0)
        r = thor.thor_grid_points(p.grid).T
        r = r / np.linalg.norm(r, axis=0)
        tau[1:4] -= (tau[1:4] * r[:, None, :]).sum(0) * r[:, None, :]
        want = dt * tau
        big = np.abs(want).max(axis=(1, 2), keepdims=True)
        assert (big[:, 0, 0] > 1e-4 * size).all()
        # the correction is formed in float32 (some 10 roundings, the projection's of the three components
        # together) and added with the storage type's rounding
        comp = np.abs(want)
        comp[1:4] = comp[1:4].sum(0)
        eps = 2.0 ** -24 if precision == thor.THOR_MIXED else 2.0 ** -53
        bound = 16 * 2.0 ** -24 * (comp + dt * np.abs(omean).reshape(5, nv, 1).max(axis=0)
                                   + dt * np.abs(tau).max(axis=(1, 2), keepdims=True)) + 2 * eps * (np.abs(a) + np.abs(b))
        assert (np.abs(a - b - want) <= bound).all(), float((np.abs(a - b - want) / bound).max())
    finally:
        p.close()
        q.close()
        thor.thor_mlp_destroy(net)
