"""The small step's p* and the float64 pressure law (thor_kernels.cuh: p_pert,
pow1p) against expm1 and log1p: both sides of every range switch, the ends of
the table, the general path, and exponents of dry air, a monatomic gas and a
nearly incompressible one."""

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
__global__ void k(Phys ph, const double* pw, const double* x, int n, double* pd, float* pf, double* e, double* l) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double th = 300.0, pi = 400.0;
  pd[i] = p_pert(ph, pi, th, x[i] * th);
  pf[i] = p_pert(ph, (float)pi, (float)th, (float)(x[i] * th));
  double a, b;
  if (!pow1p<true>(ph, pw, x[i], a, b)) {
    const double2 g = pow1p_general(x[i], ph.gamma);
    a = g.x;
    b = g.y;
  }
  e[i] = a;
  l[i] = b;
}
extern "C" int run(double gamma, const double* g, double x4, double x7, float x3, const double* pw, const double* x, int n,
                   double* pd, float* pf, double* e, double* l) {
  Phys ph;
  ph.gamma = gamma;
  ph.gamma_f = (float)gamma;
  ph.inv_gamma_f = (float)(1.0 / gamma);
  for (int i = 0; i < 7; ++i) ph.pg[i] = g[i];
  for (int i = 0; i < 3; ++i) ph.pg_f[i] = (float)g[i];
  ph.x4 = x4;
  ph.x7 = x7;
  ph.x3_f = x3;
  k<<<(n + 127) / 128, 128>>>(ph, pw, x, n, pd, pf, e, l);
  return cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("thermo")
    (d / "t.cu").write_text(CODE)
    nvcc = "/usr/local/cuda/bin/nvcc" if os.path.exists("/usr/local/cuda/bin/nvcc") else "nvcc"
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17", "--expt-relaxed-constexpr",
                    "-shared", "-Xcompiler", "-fPIC", "-I", os.path.join(ROOT, "paper_1607_05535_gb300", "csrc"),
                    str(d / "t.cu"), "-o", str(d / "t.so")], check=True)
    return ctypes.CDLL(str(d / "t.so"))


def _coefficients(gamma):
    g = [1.0]
    for k in range(1, 65):
        g.append(g[-1] * (gamma - k) / (k + 1))

    def reach(n, eps):
        for e in range(3, 60):
            if sum(abs(g[k]) * 2.0 ** (-e * k) for k in range(n + 1, 65)) <= eps:
                return 2.0 ** -e
        return 0.0

    return np.array(g[1:8]), reach(4, 2.0 ** -55), reach(7, 2.0 ** -55), reach(3, 2.0 ** -26)


@pytest.mark.parametrize("gamma", [1005.0 / 718.0, 5.0 / 3.0, 1.01])
def test_pressure_law_matches_expm1_log1p(lib, gamma):
    g, x4, x7, x3 = _coefficients(gamma)
    edges = [s * b * f for s in (1, -1) for b in (x4, x7, x3, 1.0 / 128, 1.0 / 64, 0.5, 1.0) for f in (1 - 1e-9, 1.0, 1 + 1e-9)]
    rng = np.random.default_rng(2)
    x = np.concatenate([edges, [0.0, 1e-300, -1e-12, 2.5, -0.75, -0.999], 10.0 ** rng.uniform(-12, 0.3, 4000),
                        -10.0 ** rng.uniform(-12, -0.01, 4000)])
    x = x[x > -1.0 + 1e-10]
    n = x.size
    xd = torch.tensor(x, device="cuda")
    c = 0.5 + np.arange(97) / 64.0
    pw = np.stack([c - 1, 1 / c, np.expm1(gamma * np.log1p(c - 1)), np.exp(gamma * np.log1p(c - 1)), np.log1p(c - 1), 0 * c], 1)
    pwd = torch.tensor(np.ascontiguousarray(pw), device="cuda")
    pd, e, l = (torch.empty(n, dtype=torch.float64, device="cuda") for _ in range(3))
    pf = torch.empty(n, device="cuda")
    D, P = ctypes.c_double, ctypes.c_void_p
    lib.run.argtypes = [D, P, D, D, ctypes.c_float, P, P, ctypes.c_int, P, P, P, P]
    rc = lib.run(gamma, g.ctypes.data, x4, x7, x3, pwd.data_ptr(), xd.data_ptr(), n, pd.data_ptr(), pf.data_ptr(),
                 e.data_ptr(), l.data_ptr())
    assert rc == 0
    X = x.astype(np.longdouble)
    f, ln = np.expm1(np.longdouble(gamma) * np.log1p(X)), np.log1p(X)
    rel = lambda a, b: np.max(np.abs(a.cpu().numpy() - b)[b != 0] / np.abs(b[b != 0]))
    # a handful of roundings each: x itself, the table's entries, the sum; near
    # x = -0.999 the general path loses what log1p's argument loses
    ok = np.abs(x) > 1e-290
    assert rel(pd[torch.tensor(ok)], (120000.0 / np.longdouble(gamma) * f)[ok]) < 16 * 2.0 ** -53
    assert rel(e[torch.tensor(ok)], f[ok]) < 16 * 2.0 ** -53
    assert rel(l[torch.tensor(ok)], ln[ok]) < 16 * 2.0 ** -53
    far = ok & (np.abs(x) > 1e-30) & (x > -0.99)
    xf = (x * 300.0).astype(np.float32).astype(np.longdouble) / 300
    ff = 120000.0 / np.longdouble(gamma) * np.expm1(np.longdouble(gamma) * np.log1p(xf))
    assert rel(pf[torch.tensor(far)], ff[far]) < 16 * 2.0 ** -24
    assert pd[torch.tensor(x == 0)].abs().max() == 0 and e[torch.tensor(x == 0)].abs().max() == 0
