"""The closure's features, its network over every column and its correction at
level and column counts that do not fill the 32 x 32 tiles, in both storage
precisions."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1607_05535_gb300 as thor
import workloads as wls
from harness import Pair, moving_start


def _pair(nv, precision, glevel=2):
    wl = wls.HS_G4.with_(name="closure_g%d_L%d" % (glevel, nv), glevel=glevel, nv=nv, n_large=1, noise_amp=0.5)
    p = Pair(wl, precision=precision)
    moving_start(p, p.oracle_initial())
    return p, wl


def _planes(state, nv, precision):
    """rho', M_x, M_y, M_z, (rho theta)' as stored, [5][nv][column]."""
    b = thor.thor_checkpoint_save(state)[64:].view(np.float64 if precision == thor.THOR_FP64 else np.float32)
    planes = (6 * nv + 1) * (1 if precision == thor.THOR_FP64 else 2)
    return b.reshape(planes, -1)[:5 * nv].reshape(5, nv, -1)


@pytest.mark.parametrize("precision", [thor.THOR_FP64, thor.THOR_MIXED])
@pytest.mark.parametrize("nv", [4, 12, 33])
def test_features(nv, precision):
    p, wl = _pair(nv, precision)
    try:
        rng = np.random.default_rng(1)
        mean, std = rng.standard_normal(10 * nv).astype(np.float32), rng.uniform(0.5, 2.0, 10 * nv).astype(np.float32)
        x = torch.empty((wl.ncol, 10 * nv), dtype=torch.float32, device="cuda")
        thor.thor_closure_features(p.state, torch.tensor(mean, device="cuda"), torch.tensor(std, device="cuda"), x)
        torch.cuda.synchronize()
        f = _planes(p.state, nv, precision)[:, :, :wl.ncol].astype(np.float64)
        nbr = thor.thor_grid_neighbours(p.grid)
        ok = nbr >= 0
        ring = np.where(ok, f[:, :, np.where(ok, nbr, 0)], 0.0).sum(-1) / ok.sum(1) - f
        raw = np.concatenate([f.transpose(2, 0, 1).reshape(wl.ncol, -1), ring.transpose(2, 0, 1).reshape(wl.ncol, -1)], 1)
        # each value is rounded to float32 once, then normalised in float32
        err = np.abs(x.cpu().numpy() - (raw - mean) / std)
        bound = 4 * 2.0 ** -24 * (np.abs(raw) + np.abs(mean) + np.abs((raw - mean))) / std
        assert (err <= bound).all(), (err - bound).max()
    finally:
        p.close()


@pytest.mark.parametrize("precision", [thor.THOR_FP64, thor.THOR_MIXED])
@pytest.mark.parametrize("nv", [5, 33])
def test_all_columns_at_once_match_the_batched_network(nv, precision):
    """A step with the closure on the TMA-fed pass over every column against
    the thread-staged network over batches of 50: the same bfloat16 operands,
    float32 sums in another order; a hidden value may round to the other
    bfloat16 neighbour, 2^-8 of a correction that is itself 1e-3 of the field."""
    out = []
    for tc in (1, 2):
        p, wl = _pair(nv, precision)
        net = thor.thor_mlp_create([10 * nv, 24, 40, 5 * nv], 50, seed=3)
        try:
            thor.thor_mlp_tune(net, thor.THOR_MLP_TUNE_TCGEN05, tc)
            one = lambda n, v: torch.full((n,), v, dtype=torch.float32, device="cuda")
            norm = [one(10 * nv, 0.0), one(10 * nv, 1.0), one(5 * nv, 0.0), one(5 * nv, 1e-6)]
            thor.thor_closure_attach(p.state, net, *norm, period=1)
            before = _planes(p.state, nv, precision)[:, :, :wl.ncol].astype(np.float64)
            thor.thor_step(p.state, 1, wl.n_small, 300.0)
            out.append(_planes(p.state, nv, precision)[:, :, :wl.ncol].astype(np.float64))
            thor.thor_closure_attach(p.state, None)
        finally:
            p.close()
            thor.thor_mlp_destroy(net)
    scale = np.abs(before).max(axis=(1, 2), keepdims=True)
    assert np.isfinite(out[0]).all()
    assert (np.abs(out[0] - out[1]) <= 1e-4 * scale).all(), (np.abs(out[0] - out[1]) / scale).max()
