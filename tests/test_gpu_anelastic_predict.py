"""The anelastic predictor of a float state (k_an_predict), launched by itself:
M^ = M + dt S_M is formed in float64 from the stored floats, the Cartesian S_M
from its two components and the column's basis included: 8 roundings of 2^-53
of the largest term."""

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
#include "thor_anelastic.cu"
extern "C" int run(int ncol, int nv, int colp, const float* tb, float* const* xt, float* sm2, float* zero, float* const* xo,
                   double dts, double* out) {
  using namespace thor;
  Geo<float> G{};
  G.ncol = ncol;
  G.nv = nv;
  G.colp = colp;
  G.tb = tb;
  Xf<float> X{}, O{};
  X.mx = xt[0];
  X.my = xt[1];
  X.mz = xt[2];
  X.th = X.w = zero;
  O.th = xo[0];
  O.rho = xo[1];
  Slow<float> SL{};
  SL.sm2 = sm2;
  SL.sth = SL.sw = zero;
  const size_t c = (size_t)nv * colp;
  k_an_predict<float><<<64, 256>>>(G, X, SL, O, dts, out, out + c, out + 2 * c, out + 3 * c);
  return cudaDeviceSynchronize();
}
"""


def test_slow_momentum_in_float64(tmp_path):
    (tmp_path / "t.cu").write_text(CODE)
    nvcc = "/usr/local/cuda/bin/nvcc" if os.path.exists("/usr/local/cuda/bin/nvcc") else "nvcc"
    objects = [os.path.join(ROOT, "_build", o + ".o") for o in ("grid", "thor_step", "thor_api", "thor_noalloc", "thor_mlp",
                                                                "thor_ensemble", "thor_climate")]
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17", "--expt-relaxed-constexpr",
                    "-shared", "-Xcompiler", "-fPIC,-fopenmp", "-I", os.path.join(ROOT, "paper_1607_05535_gb300", "csrc"),
                    str(tmp_path / "t.cu"), *objects, "-lgomp", "-o", str(tmp_path / "t.so")], check=True)
    lib = ctypes.CDLL(str(tmp_path / "t.so"))
    rng = np.random.default_rng(7)
    ncol, nv, colp, dts = 642, 5, 768, 300.0
    r = rng.standard_normal((3, colp))
    r /= np.linalg.norm(r, axis=0)
    s = np.where(r[2] < 0, -1.0, 1.0)
    tb = np.stack([s * r[0], s * r[1], -1.0 / (1.0 + np.abs(r[2]))]).astype(np.float32)
    m = (10.0 * rng.standard_normal((3, nv, colp))).astype(np.float32)
    sm = (0.01 * rng.standard_normal((nv, colp, 2))).astype(np.float32)
    dev = lambda a: torch.tensor(np.ascontiguousarray(a), device="cuda")
    tbd, smd, md = dev(tb), dev(sm), [dev(x) for x in m]
    zero, xo = torch.zeros((nv + 1) * colp, device="cuda"), [torch.empty(nv * colp, device="cuda") for _ in range(2)]
    out = torch.empty((4 * nv + 1) * colp, dtype=torch.float64, device="cuda")
    ptrs = lambda ts: (ctypes.c_void_p * len(ts))(*[t.data_ptr() for t in ts])
    P, I = ctypes.c_void_p, ctypes.c_int
    lib.run.argtypes = [I, I, I, P, P, P, P, P, ctypes.c_double, P]
    assert lib.run(ncol, nv, colp, tbd.data_ptr(), ptrs(md), smd.data_ptr(), zero.data_ptr(), ptrs(xo), dts, out.data_ptr()) == 0
    X, Y, A = tb.astype(np.float64)
    u, v = sm[..., 0].astype(np.float64), sm[..., 1].astype(np.float64)
    q = X * u + Y * v
    S = np.stack([u + X * A * q, v + Y * A * q, -q])
    got = out.cpu().numpy()[:3 * nv * colp].reshape(3, nv, colp)[:, :, :ncol]
    want = (m + dts * S)[:, :, :ncol]
    big = (np.abs(m) + dts * (np.abs(u) + np.abs(v)))[:, :, :ncol]
    assert (np.abs(got - want) <= 8 * 2.0 ** -53 * big).all(), float((np.abs(got - want) / big).max())
