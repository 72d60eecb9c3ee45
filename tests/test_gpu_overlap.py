"""Kernels of small float states that start while the one before drains. Only
a state on a stream of its own whose grids have at most a block per SM does
so: the same state on the default stream, and one whose block size is tuned
until its grids have more, run every kernel after the last one has ended. The
shape of a launch changes no result, so all of them agree bit for bit."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1607_05535_gb300 as thor
from harness import init_struct, planet_struct
import workloads as wls

STEPS = 6


def _checkpoint(wl, stream, tunes, **switches):
    P = wl.planet
    grid = thor.thor_grid_create(wl.glevel, wl.nv, P.radius, wl.z_top, thor.thor_spring(1.15, 1.0, 1.0, 0.01, 0.0, 10))
    state = thor.thor_state_init(grid, planet_struct(P), init_struct(wl, thor.THOR_MIXED, **switches),
                                 stream.cuda_stream if stream is not None else None)
    try:
        for knob, value in tunes:
            thor.thor_tune(state, knob, value)
        # a flow in motion: solid-body rotation with a wave, the same on every side
        r = thor.thor_grid_points(grid)
        rho, mom, w, th = (np.array(a) for a in thor.thor_state_get_all(state, wl.ncol, wl.nv))
        v = np.cross([0.0, 0.0, 1.0], r) * (20.0 + 5.0 * np.sin(4.0 * r[:, :1]))
        mom = np.ascontiguousarray(rho[..., None] * v[:, None, :])
        thor.thor_state_set_all(state, rho, mom, w, th)
        for n in (1, STEPS - 1):                         # the second call replays the graph
            thor.thor_step(state, n, wl.n_small, wl.dt)
        out = np.array(thor.thor_checkpoint_save(state))
        assert thor.thor_diag(state)["nonfinite"] == 0
        return out
    finally:
        thor.thor_state_destroy(state)
        thor.thor_grid_destroy(grid)


CASES = [
    ("held_suarez", wls.HS_G4.with_(glevel=3, nv=12, noise_amp=0.5, dt=900.0), {}),
    ("two levels more than the blocks' chunk", wls.HS_G4.with_(glevel=2, nv=28, noise_amp=0.5, dt=900.0), {}),
    ("no forcing, no hyperdiffusion", wls.HS_G4.with_(glevel=3, nv=12, noise_amp=0.5, dt=900.0, forcing="none"),
     dict(hyper=0)),
    ("no divergence damping", wls.HS_G4.with_(glevel=2, nv=9, noise_amp=0.5, dt=600.0), dict(divdamp=0)),
    ("shallow, third order", wls.HS_G4.with_(glevel=3, nv=13, noise_amp=0.5, dt=900.0), dict(shallow=1, vorder=3)),
    ("hydrostatic", wls.HS_G4.with_(glevel=3, nv=12, noise_amp=0.5, dt=900.0), dict(hydrostatic=1)),
]


@pytest.mark.parametrize("compensated", [1, 0])
@pytest.mark.parametrize("tma", [1, 0])
@pytest.mark.parametrize("name, wl, switches", CASES, ids=[c[0].replace(" ", "_") for c in CASES])
def test_early_starts_change_nothing(name, wl, switches, tma, compensated):
    tunes = [(thor.THOR_TUNE_SOLVE_TMA, tma), (thor.THOR_TUNE_COMPENSATED, compensated)]
    own = torch.cuda.Stream()
    assert -(-wl.ncol // 128) * wl.nv <= 128             # fewer than the SMs: early starts on
    early = _checkpoint(wl, own, tunes, **switches)
    for stream, more in ((None, []), (own, [(thor.THOR_TUNE_GRAPH, 0)]), (own, [(thor.THOR_TUNE_BLOCK, 32)]),
                         (own, [(thor.THOR_TUNE_BLOCK, 256)]), (own, [(thor.THOR_TUNE_ENERGY_FIXER, 0)])):
        assert np.array_equal(early, _checkpoint(wl, stream, tunes + more, **switches)), (stream, more)
