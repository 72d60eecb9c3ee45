"""The TMA-fed MLP pass at widths and batches that are no multiples of its
tiles: layers padded to multiples of 8 inside, ragged last tiles of rows and
columns, a batch of one row, split and unsplit weight gradients."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1607_05535_gb300 as thor

# Both paths multiply the same bfloat16 operands and accumulate in float32;
# a hidden value whose float32 sums fall on two sides of a bfloat16 rounding
# boundary or of zero moves by one bfloat16 spacing, 2^-8 of itself, in a few
# of the elements: 1e-3 of a result's norm.
GATE = 1e-3


def _run(sizes, m, tc, steps):
    rng = np.random.default_rng(21)
    n = sum(a * b + b for a, b in zip(sizes[:-1], sizes[1:]))
    flat = np.concatenate([np.concatenate([rng.standard_normal(a * b) / np.sqrt(a), 0.1 * rng.standard_normal(b)])
                           for a, b in zip(sizes[:-1], sizes[1:])]).astype(np.float32)
    x, t = (torch.tensor(rng.standard_normal((m, k)), dtype=torch.float32, device="cuda") for k in (sizes[0], sizes[-1]))
    net = thor.thor_mlp_create(sizes, m + 7, seed=0)
    try:
        thor.thor_mlp_tune(net, thor.THOR_MLP_TUNE_TCGEN05, tc)
        thor.thor_mlp_set_params(net, flat)
        y = torch.empty((m, sizes[-1]), device="cuda")
        g = torch.empty(n, device="cuda")
        # a larger batch first: what it left in the buffers must not show
        big = torch.ones((m + 7, sizes[0]), device="cuda")
        thor.thor_mlp_forward(net, big, torch.empty((m + 7, sizes[-1]), device="cuda"))
        thor.thor_mlp_forward(net, x, y)
        thor.thor_mlp_backward(net, t, g)
        loss = torch.zeros(1, device="cuda")
        for _ in range(steps):
            thor.thor_mlp_train_step(net, x, t, 1e-3, loss)
        p = thor.thor_mlp_get_params(net)
        return [y.cpu().numpy(), g.cpu().numpy(), p - flat, loss.cpu().numpy()]
    finally:
        thor.thor_mlp_destroy(net)


@pytest.mark.parametrize("sizes, m", [([370, 256, 256, 256, 185], 1000), ([37, 50, 19], 130), ([5, 3, 1], 1),
                                      ([9, 257, 33, 7], 33), ([200, 64, 100], 515), ([16, 24, 8], 128)])
def test_padded_pass_matches_thread_staged(sizes, m):
    for a, b in zip(_run(sizes, m, 1, 1), _run(sizes, m, 2, 1)):
        assert np.isfinite(a).all()
        assert np.linalg.norm(a - b) <= GATE * np.linalg.norm(b), (a.shape, np.linalg.norm(a - b) / np.linalg.norm(b))
