"""div_by (thor_kernels.cuh): a division by a number whose reciprocal is at
hand gives what the division gives, in both types, over the sizes it meets:
pressures by a surface pressure, sigma - sigma_b by 1 - sigma_b, Laplacians by
squared radii."""

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
template <typename R>
__global__ void k(const R* a, const R* b, int n, R* y) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) y[i] = thor::div_by(a[i], b[i], R(1) / b[i]);
}
extern "C" int run(const double* a, const double* b, int n, double* y, const float* af, const float* bf, float* yf) {
  k<<<(n + 127) / 128, 128>>>(a, b, n, y);
  k<<<(n + 127) / 128, 128>>>(af, bf, n, yf);
  return cudaDeviceSynchronize();
}
"""


def test_equals_the_division(tmp_path):
    (tmp_path / "t.cu").write_text(CODE)
    nvcc = "/usr/local/cuda/bin/nvcc" if os.path.exists("/usr/local/cuda/bin/nvcc") else "nvcc"
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17", "--expt-relaxed-constexpr",
                    "-shared", "-Xcompiler", "-fPIC", "-I", os.path.join(ROOT, "paper_1607_05535_gb300", "csrc"),
                    str(tmp_path / "t.cu"), "-o", str(tmp_path / "t.so")], check=True)
    lib = ctypes.CDLL(str(tmp_path / "t.so"))
    P = ctypes.c_void_p
    lib.run.argtypes = [P, P, ctypes.c_int, P, P, P, P]
    rng = np.random.default_rng(8)
    n = 1 << 20
    sign = rng.choice([-1.0, 1.0], n)
    parts = [(rng.uniform(1e2, 1.1e5, n), rng.uniform(8e4, 2.3e7, n)),                    # p / p_s
             (rng.uniform(-0.7, 0.4, n), np.full(n, 1.0 - 0.7)), (rng.uniform(-0.2, 1.0, n), np.full(n, 2.0 * (1.0 - 0.12))),
             (sign * 10.0 ** rng.uniform(-12, 12, n), rng.uniform(6.3e6, 1.1e8, n) ** 2)]  # lap / r^2
    a, b = (np.concatenate(x) for x in zip(*parts))
    a[:3] = 0.0
    dev = lambda x: torch.tensor(x, device="cuda")
    ad, bd, af, bf = dev(a), dev(b), dev(a.astype(np.float32)), dev(b.astype(np.float32))
    y, yf = torch.empty_like(ad), torch.empty_like(af)
    assert lib.run(ad.data_ptr(), bd.data_ptr(), a.size, y.data_ptr(), af.data_ptr(), bf.data_ptr(), yf.data_ptr()) == 0
    assert np.array_equal(y.cpu().numpy(), a / b)
    assert np.array_equal(yf.cpu().numpy(), a.astype(np.float32) / b.astype(np.float32))
