"""The gradient of the small step's one scalar in float states (k_ss_mom),
launched by itself on a table of seven-point stencils whose weights add up to
zero, as a gradient's do. The values carry a large common part; the result's
error stays on the scale of their differences:
each term w_j (v_j - mean) is rounded in the weight, the difference and the
product's sum, at most 10 roundings of 2^-24 of sum |w_j| |v_j - mean|."""

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
#include "thor_step.cu"
extern "C" int run(int ncol, int nv, int colp, const int* nbr, const float* wg2, const float* inv_rc, float* p, float* sm2,
                   float* m2) {
  using namespace thor;
  Geo<float> G{};
  G.ncol = ncol;
  G.nv = nv;
  G.colp = colp;
  G.nbr = nbr;
  G.wg2 = wg2;
  VR<float> U{};
  U.inv_rc = inv_rc;
  Slow<float> SL{};
  SL.sm2 = sm2;
  Pert<float> P{};
  P.p = p;
  P.m2 = m2;
  const Xf<float> X{};
  k_ss_mom<float, false><<<dim3((ncol + 127) / 128, nv), 128>>>(G, U, SL, P, Work<float>{}, 1.0f, 0, X, X, X, X, 1, 0, nv);
  return cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("gradient")
    (d / "t.cu").write_text(CODE)
    nvcc = "/usr/local/cuda/bin/nvcc" if os.path.exists("/usr/local/cuda/bin/nvcc") else "nvcc"
    objects = [os.path.join(ROOT, "_build", o + ".o") for o in ("grid", "thor_api", "thor_noalloc", "thor_mlp", "thor_ensemble",
                                                                "thor_climate", "thor_anelastic")]
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17", "--expt-relaxed-constexpr",
                    "-shared", "-Xcompiler", "-fPIC,-fopenmp", "-I", os.path.join(ROOT, "paper_1607_05535_gb300", "csrc"),
                    str(d / "t.cu"), *objects, "-lgomp", "-o", str(d / "t.so")], check=True)
    return ctypes.CDLL(str(d / "t.so"))


@pytest.mark.parametrize("common", [0.0, 1.0, 1.0e3, -1.0e5])
def test_error_scales_with_the_differences(lib, common):
    rng = np.random.default_rng(3)
    ncol, nv, colp = 1000, 3, 1024
    nbr = rng.integers(0, ncol, (6, colp)).astype(np.int32)
    nbr[5, :12] = np.arange(12)                                  # pentagons: the point itself, weight zero
    w = rng.standard_normal((7, colp, 2))
    w[6, :12] = 0.0
    w[0] = -w[1:].sum(0)
    v = (common + rng.standard_normal((nv, colp))).astype(np.float32)
    wf = w.astype(np.float32)
    n = np.concatenate([np.arange(colp)[None], nbr])
    n[:, ncol:] = 0
    dev = lambda a: torch.tensor(np.ascontiguousarray(a), device="cuda")
    m2 = torch.zeros((nv, colp, 2), device="cuda")
    sm2 = torch.zeros_like(m2)
    args = [dev(n[1:].astype(np.int32)), dev(wf), torch.ones(nv, device="cuda"), dev(v), sm2, m2]
    P, I = ctypes.c_void_p, ctypes.c_int
    lib.run.argtypes = [I, I, I] + [P] * 6
    assert lib.run(ncol, nv, colp, *[a.data_ptr() for a in args]) == 0
    got = -m2.cpu().numpy()[:, :ncol].astype(np.float64)
    near = v.astype(np.float64)[:, n]                            # [nv][7][colp]
    exact = np.einsum("jca,kjc->kca", w, near)[:, :ncol]
    off = np.abs(near - near.mean(1, keepdims=True))
    # and the float mean is a multiple of 1 / 7 rounded: what it leaves over is common to all seven
    bound = 10 * 2.0 ** -24 * (np.einsum("jca,kjc->kca", np.abs(w), off) + 2.0 ** -22 * abs(common) * np.abs(w).sum(0))[:, :ncol]
    assert (np.abs(got - exact) <= bound).all(), float((np.abs(got - exact) / bound).max())
