"""Mixed-precision members stepped in an ensemble and alone: the same device
code, with the contraction of the one cancelling difference that feeds the
hyperdiffusion (T' = T - T_bar) written out, so that both round alike. Deep
nonhydrostatic Held-Suarez members of several grids, planets and time steps
agree bit for bit after two large steps, low parts included."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1607_05535_gb300 as thor
from harness import planet_struct
import workloads as wls


def test_members_round_as_alone():
    nv, stream = 20, torch.cuda.Stream()
    grids, pairs = [], []
    members = wls.ensemble_members(6, n_small=8)
    try:
        for i, m in enumerate(members):
            P = m.planet
            grids.append(thor.thor_grid_create(m.glevel, nv, P.radius, wls.ENSEMBLE_Z_TOP,
                                               thor.thor_spring(1.15, 1.0, 1.0, 0.01, 0.0, 10)))
            init = thor.thor_init(300.0, 1.0e5, 0.5, 50 + i, thor.THOR_FORCING_HELD_SUAREZ, 300.0, thor.THOR_MIXED, 1, 1)
            pairs.append([thor.thor_state_init(grids[-1], planet_struct(P), init, stream.cuda_stream) for _ in range(2)])
        ens = thor.thor_ensemble_create([a for a, _ in pairs], stream.cuda_stream)
        try:
            thor.thor_ensemble_step(ens, 2, [m.n_small for m in members], [m.dt for m in members])
            for (a, b), m in zip(pairs, members):
                thor.thor_step(b, 2, m.n_small, m.dt)
                assert np.array_equal(thor.thor_checkpoint_save(a), thor.thor_checkpoint_save(b)), m
        finally:
            thor.thor_ensemble_destroy(ens)
    finally:
        for pair in pairs:
            for s in pair:
                thor.thor_state_destroy(s)
        for g in grids:
            thor.thor_grid_destroy(g)
