"""Networks created by several threads of a fresh process at once all find the
tensor-map encoder: their launches of one forward pass are the TMA-fed ones
(the thread-staged path would give other bits at a width that is a multiple
of 8 with split sums, and keeps no transposed inputs for the backward pass), so
gradients agree with a network created alone, bit for bit."""

import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

CODE = r"""
import threading
import numpy as np
import torch
import paper_1607_05535_gb300 as thor

torch.cuda.init()
torch.zeros(1, device="cuda")
sizes, m, n = [320, 256, 160], 1024, 8
g = torch.Generator("cuda").manual_seed(1)
x, t = (torch.randn(m, k, generator=g, device="cuda") for k in (320, 160))
nets, gate = [None] * n, threading.Barrier(n)

def make(i):
    torch.cuda.set_device(0)
    gate.wait()
    nets[i] = thor.thor_mlp_create(sizes, m, seed=3)

threads = [threading.Thread(target=make, args=(i,)) for i in range(n)]
[h.start() for h in threads]
[h.join() for h in threads]
nets.append(thor.thor_mlp_create(sizes, m, seed=3))
out = []
for net in nets:
    y, grad = torch.empty(m, 160, device="cuda"), torch.empty(thor.thor_mlp_info(net), device="cuda")
    thor.thor_mlp_forward(net, x, y)
    thor.thor_mlp_backward(net, t, grad)
    out.append((y.cpu().numpy(), grad.cpu().numpy()))
for a in out:
    assert np.array_equal(a[0], out[-1][0]) and np.array_equal(a[1], out[-1][1])
print("same")
"""


def test_concurrent_creation():
    r = subprocess.run([sys.executable, "-c", CODE], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.strip() == "same", r.stdout + r.stderr
