"""A network with a width that is no multiple of 8 adds up its gradients in the
same order on the TMA-fed and the thread-staged path: outputs, gradients and
the weights after a few Adam steps (which would amplify any difference of
rounding) are equal bit for bit, at ragged tiles of rows and columns."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from test_gpu_mlp_widths import _run


@pytest.mark.parametrize("sizes, m", [([370, 256, 256, 256, 185], 1000), ([37, 50, 19], 130), ([9, 257, 33, 7], 33),
                                      ([200, 64, 100], 515), ([5, 3, 1], 1)])
def test_both_paths_give_the_same_weights(sizes, m):
    for what, a, b in zip(("outputs", "gradients", "weights"), _run(sizes, m, 1, 4), _run(sizes, m, 2, 4)):
        assert np.array_equal(a, b), (what, np.abs(a - b).max())
