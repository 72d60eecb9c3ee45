"""The loss a training step reports: the mean square of forward output minus
target, its partial sums (one per tile of the output) added in float32: n / 2
roundings of a sum of positive terms at worst, far fewer by tiles and trees;
the bound takes the square root of n."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1607_05535_gb300 as thor


@pytest.mark.parametrize("tc", [0, 1, 2])
@pytest.mark.parametrize("sizes, m", [([320, 256, 160], 1024), ([37, 50, 19], 130), ([16, 8], 1), ([24, 40, 8], 129)])
def test_loss_is_the_mean_square(sizes, m, tc):
    g = torch.Generator("cuda").manual_seed(2)
    x, t = (torch.randn(m, k, generator=g, device="cuda") for k in (sizes[0], sizes[-1]))
    net = thor.thor_mlp_create(sizes, m, seed=4)
    try:
        thor.thor_mlp_tune(net, thor.THOR_MLP_TUNE_TCGEN05, tc)
        y, loss = torch.empty(m, sizes[-1], device="cuda"), torch.zeros(1, device="cuda")
        thor.thor_mlp_forward(net, x, y)
        thor.thor_mlp_train_step(net, x, t, 1e-3, loss)
        d = y.double().cpu().numpy() - t.double().cpu().numpy()
        want = float(np.mean(d * d))
        assert abs(float(loss) - want) <= (4 + np.sqrt(d.size)) * 2.0 ** -24 * want
    finally:
        thor.thor_mlp_destroy(net)
