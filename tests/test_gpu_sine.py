"""The day-night profile's sine (thor_kernels.cuh: rsinpi) of float states is
evaluated in float64 and rounded once: at most half a unit in the last place
from sin(pi x), over the range of (sigma - sigma_s) / (2 (1 - sigma_s))."""

import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CODE = r"""
#include "thor_kernels.cuh"
__global__ void k(const float* x, int n, float* y) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) y[i] = thor::rsinpi<float>(x[i]);
}
extern "C" int run(const float* x, int n, float* y) {
  k<<<(n + 127) / 128, 128>>>(x, n, y);
  return cudaDeviceSynchronize();
}
"""


def test_sine_is_rounded_once(tmp_path):
    (tmp_path / "t.cu").write_text(CODE)
    nvcc = "/usr/local/cuda/bin/nvcc" if os.path.exists("/usr/local/cuda/bin/nvcc") else "nvcc"
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17", "--expt-relaxed-constexpr",
                    "-shared", "-Xcompiler", "-fPIC", "-I", os.path.join(ROOT, "paper_1607_05535_gb300", "csrc"),
                    str(tmp_path / "t.cu"), "-o", str(tmp_path / "t.so")], check=True)
    lib = ctypes.CDLL(str(tmp_path / "t.so"))
    lib.run.argtypes = [ctypes.c_void_p, ctypes.c_int, ctypes.c_void_p]
    rng = np.random.default_rng(4)
    x = np.concatenate([rng.uniform(-0.07, 0.6, 1 << 20), 10.0 ** rng.uniform(-8, -1, 1 << 16)]).astype(np.float32)
    xd = torch.tensor(x, device="cuda")
    y = torch.empty_like(xd)
    assert lib.run(xd.data_ptr(), x.size, y.data_ptr()) == 0
    exact = np.sin(np.longdouble("3.14159265358979323846264338327950288") * x.astype(np.longdouble))
    ulp = np.spacing(np.abs(exact).astype(np.float32)).astype(np.longdouble)
    err = np.abs(y.cpu().numpy() - exact) / ulp
    # half a unit, and the float64 value's own last place (2^-28 of a float32 unit, taken 16 times)
    assert err.max() <= 0.5 + 2.0 ** -24, float(err.max())
