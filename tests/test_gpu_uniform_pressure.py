"""A horizontally uniform, hydrostatically balanced state far from the
reference column has no horizontal pressure gradient. In float states its
discrete gradient is taken by differences, so the momentum that a planet
without rotation picks up from rest stays far below one rounding of p' at a
grid distance, which is what a sum of weights times p' leaves: bounded by a
twentieth of 2^-24 p' / dx over the run."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1607_05535_gb300 as thor


@pytest.mark.parametrize("switches", [dict(), dict(shallow=1), dict(vorder=3), dict(hydrostatic=1)])
@pytest.mark.parametrize("glevel", [3, 5])
def test_no_wind_from_a_uniform_pressure(glevel, switches):
    nv, radius, steps, dt = 12, 6.371e6, 4, 600.0
    grid = thor.thor_grid_create(glevel, nv, radius, 30.0e3, thor.thor_spring(1.15, 1.0, 1.0, 0.01, 0.0, 10))
    n = 10 * 4 ** glevel + 2
    planet = thor.thor_planet(radius, 0.0, 9.8, 287.0, 1005.0, 1.0e5, 0.005)

    def state(T):
        init = thor.thor_init(T, 1.0e5, 0.0, 1, thor.THOR_FORCING_NONE, 300.0, thor.THOR_MIXED, 0, 1,
                              switches.get("shallow", 0), switches.get("hydrostatic", 0), 0, switches.get("vorder", 1))
        return thor.thor_state_init(grid, planet, init, None)

    warm, s = state(330.0), state(280.0)
    try:
        rho, mom, w, th = (np.array(a) for a in thor.thor_state_get_all(warm, n, nv))
        ref = thor.thor_state_get_all(s, n, nv)
        thor.thor_state_set_all(s, rho, np.zeros_like(mom), np.zeros_like(w), th)
        eos = lambda t: 1.0e5 * (287.0 * t / 1.0e5) ** (1005.0 / (1005.0 - 287.0))
        dp = np.abs(eos(th) - eos(np.array(ref[3]))).max()
        assert dp > 3.0e3
        thor.thor_step(s, steps, 8, dt)
        got = np.abs(np.array(thor.thor_state_get_all(s, n, nv)[1])).max()
        dx = np.sqrt(2.0 * np.pi / 5.0) * radius / 2 ** glevel
        assert got <= 0.05 * 2.0 ** -24 * dp / dx * steps * dt, (got, 2.0 ** -24 * dp / dx * steps * dt)
    finally:
        for x in (warm, s):
            thor.thor_state_destroy(x)
        thor.thor_grid_destroy(grid)
