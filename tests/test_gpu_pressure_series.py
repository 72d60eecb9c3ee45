"""The float p* of the small step (thor_kernels.cuh: p_pert) for given Pi, Th
and Th*: two roundings (Pi Th*, the final sum), the polynomial's and the
quotient's own errors times gamma - 1 and x, in all at most 2.5 units of 2^-24
of the result for |x| up to 1/24, more than a large step reaches; beyond the
series' range the general functions on Pi Th / gamma, 12 units."""

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
using namespace thor;
__global__ void k(Phys ph, const float* pi, const float* th, const float* d, int n, float* p) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) p[i] = p_pert(ph, pi[i], th[i], d[i]);
}
extern "C" int run(double gamma, const double* g, float x3, const float* pi, const float* th, const float* d,
                   int n, float* p) {
  Phys ph;
  ph.gamma = gamma;
  ph.gamma_f = (float)gamma;
  ph.inv_gamma_f = (float)(1.0 / gamma);
  for (int i = 0; i < 4; ++i) ph.pg_f[i] = (float)g[i];
  ph.x3_f = x3;
  k<<<(n + 127) / 128, 128>>>(ph, pi, th, d, n, p);
  return cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("series")
    (d / "t.cu").write_text(CODE)
    nvcc = "/usr/local/cuda/bin/nvcc" if os.path.exists("/usr/local/cuda/bin/nvcc") else "nvcc"
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17", "--expt-relaxed-constexpr",
                    "-shared", "-Xcompiler", "-fPIC", "-I", os.path.join(ROOT, "paper_1607_05535_gb300", "csrc"),
                    str(d / "t.cu"), "-o", str(d / "t.so")], check=True)
    return ctypes.CDLL(str(d / "t.so"))


@pytest.mark.parametrize("gamma", [1005.0 / 718.0, 13226.5 / (13226.5 - 3779.0), 5.0 / 3.0])
def test_rounding(lib, gamma):
    g = [1.0]
    for k in range(1, 65):
        g.append(g[-1] * (gamma - k) / (k + 1))

    def reach(n):
        for e in range(48, 960):
            if sum(abs(g[k]) * 2.0 ** (-e * k / 16) for k in range(n + 1, 65)) <= 2.0 ** -26:
                return 2.0 ** (-e / 16)
        return 0.0

    c, x3 = np.array(g[1:5]), float(np.float32(reach(4)))
    assert x3 >= 1.0 / 24
    rng = np.random.default_rng(6)
    n = 1 << 20
    x = rng.choice([-1.0, 1.0], n) * 10.0 ** rng.uniform(-8, -0.4, n)
    x[:6] = [x3, -x3, 1.001 * x3, -1.001 * x3, 0.0, 1e-30]
    th = (10.0 ** rng.uniform(-2, 3, n)).astype(np.float32)
    pi = (10.0 ** rng.uniform(1, 3, n)).astype(np.float32)
    d = (x * th).astype(np.float32)
    dev = [torch.tensor(a, device="cuda") for a in (pi, th, d)]
    out = torch.empty(n, device="cuda")
    F, P = ctypes.c_float, ctypes.c_void_p
    lib.run.argtypes = [ctypes.c_double, P, F, P, P, P, ctypes.c_int, P]
    assert lib.run(gamma, c.ctypes.data, x3, *[a.data_ptr() for a in dev], n, out.data_ptr()) == 0
    q = d.astype(np.longdouble) / th
    G = np.longdouble(gamma)
    exact = pi * th.astype(np.longdouble) / G * np.expm1(G * np.log1p(q))
    nz = exact != 0
    err = np.abs(out.cpu().numpy() - exact)[nz] / np.abs(exact[nz]) * 2.0 ** 24
    small = np.abs(q[nz]) <= 1.0 / 24
    assert err[small].max() <= 2.5, float(err[small].max())
    assert err.max() <= 12.0, float(err.max())
    assert not out.cpu().numpy()[~nz].any()
