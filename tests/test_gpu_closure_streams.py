"""One network attached to two states on two streams: each state's evaluation
follows its own features and comes before its own correction, whatever is
queued on the other stream, and training on one stream is ordered against the
evaluations on the other. The same calls with a wait after each give the
reference; the results are equal bit for bit."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1607_05535_gb300 as thor
from harness import init_struct, planet_struct
import workloads as wls

WL = wls.HS_G4.with_(name="hs_g3_L12", glevel=3, nv=12, noise_amp=0.5)
DELAY = 100_000_000      # cycles, about 50 ms


def _run(tc, wait):
    """Fields of both states after two steps each, a training step between."""
    nv, P = WL.nv, WL.planet
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    grid = thor.thor_grid_create(WL.glevel, nv, P.radius, WL.z_top, thor.thor_spring(1.15, 1.0, 1.0, 0.01, 0.0, 10))
    net = thor.thor_mlp_create([10 * nv, 48, 5 * nv], 200, seed=3, stream=streams[0].cuda_stream)
    states = [thor.thor_state_init(grid, planet_struct(P), init_struct(WL.with_(seed=9 + i), thor.THOR_MIXED),
                                   s.cuda_stream) for i, s in enumerate(streams)]
    try:
        thor.thor_mlp_tune(net, thor.THOR_MLP_TUNE_TCGEN05, tc)
        g = torch.Generator("cuda").manual_seed(1)
        x, t = (torch.randn(200, n, generator=g, device="cuda") for n in (10 * nv, 5 * nv))
        one = lambda n, v: torch.full((n,), v, dtype=torch.float32, device="cuda")
        norm = [one(10 * nv, 0.0), one(10 * nv, 0.05), one(5 * nv, 0.0), one(5 * nv, 1e-7)]
        torch.cuda.synchronize()
        for s in states:
            thor.thor_closure_attach(s, net, *norm, period=1)      # the network is on the second stream from here

        def then(stream=None):
            if wait:
                torch.cuda.synchronize()
            elif stream is not None:                               # what follows on this stream comes late
                with torch.cuda.stream(streams[stream]):
                    torch.cuda._sleep(DELAY)

        then(1)
        thor.thor_step(states[0], 1, WL.n_small, 300.0)
        then()
        thor.thor_step(states[1], 1, WL.n_small, 300.0)
        then(0)
        thor.thor_step(states[0], 1, WL.n_small, 300.0)            # reads the weights late
        then()
        thor.thor_mlp_train_step(net, x, t, 1e-2)
        then(1)
        thor.thor_mlp_train_step(net, x, t, 1e-2)                  # changes them late
        then()
        for s in states:
            thor.thor_step(s, 1, WL.n_small, 300.0)
            then()
        torch.cuda.synchronize()
        out = [np.array(thor.thor_checkpoint_save(s)) for s in states] + [thor.thor_mlp_get_params(net)]
        for s in states:
            thor.thor_closure_attach(s, None)
        return out
    finally:
        for s in states:
            thor.thor_state_destroy(s)
        thor.thor_mlp_destroy(net)
        thor.thor_grid_destroy(grid)


@pytest.mark.parametrize("tc", [1, 2])
def test_one_network_two_streams(tc):
    ref = _run(tc, True)
    for a, b in zip(_run(tc, False), ref):
        assert np.array_equal(a, b)
    again = _run(tc, True)                                         # the reference itself repeats
    assert all(np.array_equal(a, b) for a, b in zip(again, ref))


def test_network_outlives_a_state_and_its_stream():
    """The network stays usable on a state attached earlier, and on one
    attached after the last state is gone."""
    nv, P = WL.nv, WL.planet
    sp = thor.thor_spring(1.15, 1.0, 1.0, 0.01, 0.0, 10)
    grid = thor.thor_grid_create(WL.glevel, nv, P.radius, WL.z_top, sp)
    net = thor.thor_mlp_create([10 * nv, 48, 5 * nv], 200, seed=3)
    one = lambda n, v: torch.full((n,), v, dtype=torch.float32, device="cuda")
    norm = [one(10 * nv, 0.0), one(10 * nv, 0.05), one(5 * nv, 0.0), one(5 * nv, 1e-7)]
    out = []
    streams = [torch.cuda.Stream() for _ in range(2)]
    try:
        for s in streams:
            state = thor.thor_state_init(grid, planet_struct(P), init_struct(WL, thor.THOR_MIXED), s.cuda_stream)
            thor.thor_closure_attach(state, net, *norm, period=1)
            thor.thor_step(state, 2, WL.n_small, 300.0)
            out.append(np.array(thor.thor_checkpoint_save(state)))
            thor.thor_state_destroy(state)
        assert np.array_equal(*out)
    finally:
        thor.thor_mlp_destroy(net)
        thor.thor_grid_destroy(grid)
