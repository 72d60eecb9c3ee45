"""Attaching a closure takes the output and two bfloat16 buffers of the widest
layer per column, no float32 features beside them, and detaching gives them
back."""

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1607_05535_gb300 as thor
from harness import init_struct, planet_struct
import workloads as wls


def test_attached_bytes():
    wl = wls.HS_G6.with_(glevel=6, nv=32)
    P, nv = wl.planet, wl.nv
    grid = thor.thor_grid_create(wl.glevel, nv, P.radius, wl.z_top, thor.thor_spring(1.15, 1.0, 1.0, 0.01, 0.0, 10))
    state = thor.thor_state_init(grid, planet_struct(P), init_struct(wl, thor.THOR_MIXED), None)
    net = thor.thor_mlp_create([10 * nv, 256, 5 * nv], 1024, seed=1)
    try:
        one = lambda n: torch.ones(n, device="cuda")
        norm = [one(10 * nv), one(10 * nv), one(5 * nv), one(5 * nv)]
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        thor.thor_closure_attach(state, net, *norm, period=1)
        torch.cuda.synchronize()
        used = free - torch.cuda.mem_get_info()[0]
        need = wl.ncol * (5 * nv * 4 + 2 * 10 * nv * 2)
        assert used <= need + (8 << 20), (used, need)             # pages of 2 MB, a few events
        thor.thor_closure_attach(state, None)
        torch.cuda.synchronize()
        assert free - torch.cuda.mem_get_info()[0] <= 8 << 20
    finally:
        thor.thor_state_destroy(state)
        thor.thor_mlp_destroy(net)
        thor.thor_grid_destroy(grid)
