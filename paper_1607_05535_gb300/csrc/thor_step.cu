// Kernels of one large step (Sec. 3-5 of Mendonca et al. 2016) and their
// launch sequence.
//
// Stencil kernels: one thread per column, looping over a chunk of levels, so
// the per-column stencil weights are loaded once per chunk; the block's
// second index picks the chunk. A warp covers 32 consecutive columns of one
// level, so every field access is a coalesced (or neighbour-shifted) row of
// one plane.
//
// The vertical solve is split: k_ss_flux (a stencil kernel like the others)
// forms the per-cell parts of the column equations, and k_ss_solve runs the
// tridiagonal elimination from both ends: two sweeping warps per 32 columns in
// float storage, the two halves of one warp per 16 columns in float64.
#include "../../include/thor.h"
#include "thor_impl.cuh"
#include "thor_reduce.cuh"

#include <utility>

namespace thor {

// ---------------------------------------------------------------- launch helper

template <typename... K, typename... A>
cudaError_t launch_k(void (*kern)(K...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, A&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  return cudaLaunchKernelEx(&cfg, kern, std::forward<A>(args)...);
}
template <typename... K, typename... A>
cudaError_t launch_hint(LaunchHint hint, void (*kern)(K...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                        A&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[2];
  int n = 0;
  if (hint.after) {
    at[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[n++].val.programmaticStreamSerializationAllowed = 1;
  }
  if (hint.carveout >= 0) {
    at[n].id = cudaLaunchAttributePreferredSharedMemoryCarveout;
    at[n++].val.sharedMemCarveout = (unsigned)hint.carveout;
  }
  cfg.attrs = at;
  cfg.numAttrs = n;
  return cudaLaunchKernelEx(&cfg, kern, std::forward<A>(args)...);
}

// Each step of the method is a device function over one block of columns
// (block indices passed in); the kernels below run it either for one state
// (block indices from the launch grid) or for a whole ensemble of states in
// one launch (block -> (member, local block) from a block map).


// ---------------------------------------------------------------- slow terms

// Pointwise derived quantities at the stage state: p', Pi = gamma p / rho theta,
// T', theta, the full
// 3-D velocity, v_h = M/rho (centres) and v_r = W/rho (interfaces); the
// velocities go into packed planes with theta (v4) and T' (vh4) beside them,
// the fields the next stencils gather together.
// HO: the order-k interpolation of the explicit terms (thor_init.vorder > 1)
template <typename R, bool HO = false>
__device__ __forceinline__ void d_derived(const Geo<R>& G, const VR<R>& U, const Phys& ph, const Xf<R>& X, const Work<R>& T, R* pi, int shallow, int kchunk,
                                          int bx, int by) {
  int c = bx * blockDim.x + threadIdx.x;
  pdl_next();
  if (c >= G.ncol) return;
  const R gamma = pc<R>(ph.gamma, ph.gamma_f), inv_Rd = pc<R>(ph.inv_Rd, ph.inv_Rd_f);
  R rx = ld(G.rhat + (c)), ry = ld(G.rhat + (G.colp + c)), rz = ld(G.rhat + (2 * G.colp + c));
  const int S = pdl_wait(G.colp);
  int k0 = by * kchunk, k1 = min(G.nv + 1, k0 + kchunk);
#pragma unroll 2
  for (int k = k0; k < k1; ++k) {
    if (k < G.nv) {
      int i = k * S + c;
      R rho = ld(U.rhob + (k)) + ld(X.rho + (i));
      R thp = ld(X.th + (i));
      R pp = eos_level(U, ph, k, thp);
      R p = ld(U.pb + (k)) + pp;
      R inv = R(1) / rho;
      R wc = HO ? vint_centre(U, X.w, k, c, S, G.nv)
                           : ld(U.clo + (k)) * ld(X.w + (i)) + ld(U.chi + (k)) * ld(X.w + (i + S));
      R mx = ld(X.mx + (i)), my = ld(X.my + (i)), mz = ld(X.mz + (i));
      const R thfull = ld(U.thb + (k)) + thp;
      const R theta = thfull * inv;
      T.pp[i] = pp;
      pi[i] = gamma * p / thfull;
      T.theta[i] = theta;
      st4(T.v4, i, (mx + wc * rx) * inv, (my + wc * ry) * inv, (mz + wc * rz) * inv, theta);
      // T' = p / (rho Rd) - T_bar in one rounding of the difference, written out: left to
      // contraction, the ensemble's kernel rounded T first, which as noise of 2^-25 of
      // 300 K went through the hyperdiffusion (error of rho' after a step +11%)
      st4(T.vh4, i, mx * inv, my * inv, mz * inv, fmar<R>(p * inv, inv_Rd, -ld(U.Tb + (k))));
      if (shallow) T.wc[i] = wc * inv;
    }
    if (k >= 1 && k < G.nv) {
      int i = k * S + c;
      R rlo = ld(U.rhob + (k - 1)) + ld(X.rho + (i - S)), rhi = ld(U.rhob + (k)) + ld(X.rho + (i));
      if constexpr (HO)
        T.vr[i] = ld(X.w + (i)) / vint_iface(U, X.rho, U.rhob, k, c, S, G.nv);
      else
        T.vr[i] = ld(X.w + (i)) / (ld(U.wlo + (k)) * rlo + ld(U.whi + (k)) * rhi);
    } else if (k == 0 || k == G.nv) {
      T.vr[k * S + c] = 0;
    }
  }
}

// First Laplacians of the hyperdiffusion (Sec. 4), already multiplied by
// K_d and, for the momentum and temperature terms, by rho.
template <typename R, bool HO = false>
__device__ __forceinline__ void d_lap1(const Geo<R>& G, const VR<R>& U, const Xf<R>& X, const Work<R>& T, R Kd, int kchunk, int bx, int by,
                                       int kend) {
  int c = bx * blockDim.x + threadIdx.x;
  pdl_next();
  if (c >= G.ncol) return;
  Nbr7 nb = load_nbr(G, c);
  W7<R> wl = load_w7(G.wlap, G.colp, c);
  const int S = pdl_wait(G.colp);
  int k0 = by * kchunk, k1 = min(kend, k0 + kchunk);
#pragma unroll 2
  for (int k = k0; k < k1; ++k) {
    if (k < G.nv) {
      int o = k * S;
      R inv_r2 = ld(U.inv_rc2 + (k));
      R rho = ld(U.rhob + (k)) + ld(X.rho + (o + c));
      R rk = rho * Kd * inv_r2;
      const Q4<R> lv = apply7x4(wl, nb, T.vh4, o);       // lap of v_h (x, y, z) and of T'
      st4(T.q4, o + c, rk * lv.x, rk * lv.y, rk * lv.z, Kd * apply7(wl, nb, X.rho + o) * inv_r2);
      T.qT[o + c] = rk * lv.w;
    }
    if (k >= 1 && k < G.nv) {
      int o = k * S;
      R rlo = ld(U.rhob + (k - 1)) + ld(X.rho + (o - S + c)), rhi = ld(U.rhob + (k)) + ld(X.rho + (o + c));
      R rif = HO ? vint_iface(U, X.rho, U.rhob, k, c, S, G.nv) : ld(U.wlo + (k)) * rlo + ld(U.whi + (k)) * rhi;
      T.qvr[o + c] = div_by(rif * Kd * apply7(wl, nb, T.vr + o), ld(U.ri2 + (k)), ld(U.inv_ri2 + (k)));
    } else if (k == 0 || k == G.nv) {
      T.qvr[k * S + c] = 0;
    }
  }
}

// Slow tendencies at the centres (right-hand sides of Eqs. mom2, dens2, pt2):
// S_M = -grad_h p - A_h - C_h + F_M, S_rho = -div(M) - div(W) + F_rho,
// S_th = F_th - div(theta M) - div(theta W), plus Dsc = div(M) + div(W) of the
// stage state (divergence damping) and the radial advection+Coriolis. In the first stage (stage state = X^t) Dsc is also
// kept in d0: it is the divergence D that the first small step of every
// stage damps, since there M^(s) + M* = M^t and W^(s) + W* = W^t.
// SH: the shallow-atmosphere approximation of Sec. 3 (r = A in the tables;
// here the traditional Coriolis, 2 Omega sin(lat) r x M on the horizontal
// momentum only, and the horizontal velocity and w advected without the
// metric terms the approximation drops)
// DENSE: one level at a time in few registers, for more threads in flight
// (k_slow chooses)
template <typename R, bool SH = false, bool HO = false, bool DENSE = false>
__device__ __forceinline__ void d_slow(const Geo<R>& G, const VR<R>& U, const Phys& ph, const Xf<R>& X, const Work<R>& T, const Slow<R>& SL, int hyper,
                                            R* d0, int kchunk, int bx, int by, int kend) {
  int c = bx * blockDim.x + threadIdx.x;
  pdl_next();
  if (c >= G.ncol) return;
  const int S0 = G.colp;
  Nbr7 nb = load_nbr(G, c);
  // the divergence and Laplacian weights; the gradient of p below is taken
  // with the divergence weights plus the centre correction, unprojected
  // (S_M is projected as a whole). A constant has no tangential gradient, so float
  // states take the differences to the centre, whose products round on the scale of
  // the differences; the centre's own weights drop out
  constexpr bool kByDifference = sizeof(R) == sizeof(float);
  W7x3<R> wd;
  W7<R> wl;
  load_w7x3_lap(G.wdiv, S0, c, wd, wl);
  const R gcx = ld(G.gcor + (c)), gcy = ld(G.gcor + (S0 + c)), gcz = ld(G.gcor + (2 * S0 + c));
  R rx = ld(G.rhat + (c)), ry = ld(G.rhat + (S0 + c)), rz = ld(G.rhat + (2 * S0 + c));
  const R tA = ld(G.tb + (2 * S0 + c));
  const R two_om = pc<R>(ph.two_omega, ph.two_omega_f), Rd = pc<R>(ph.Rd, ph.Rd_f);
  const int S = pdl_wait(G.colp);
  int k0 = by * kchunk, k1 = min(kend, k0 + kchunk);
  constexpr int kUnroll = sizeof(R) == sizeof(float) && !DENSE ? 2 : 1;   // float64: registers
#pragma unroll kUnroll
  for (int k = k0; k < k1; ++k) {
    const int o = k * S, i = o + c;
    const R inv_r = ld(U.inv_rc + (k)), inv_r2 = ld(U.inv_rc2 + (k));
    const R sql = ld(U.sq_lo + (k)), sqh = ld(U.sq_hi + (k));
    // one pass over the 7-point neighbourhood, each neighbour value loaded
    // once: the edge flux f = w . M of the momentum (shared by the continuity,
    // advection and rho-theta divergences), the pressure gradient and the
    // second Laplacians of the hyperdiffusion
    R sa0 = 0, sa1 = 0, sa2 = 0, sa3 = 0, sdh = 0, sdt = 0, gx = 0, gy = 0, gz = 0;
    R hr = 0, hx = 0, hy = 0, hz = 0, hT = 0, p0 = 0;
    // advected velocity (packed with theta or T'): the full 3-D one, or (SH)
    // the horizontal one and w
    const R* av4 = SH ? T.vh4 : T.v4;
#pragma unroll
    for (int j = 0; j < 7; ++j) {
      const int q = o + nb.n[j];
      const R f = wd.x[j] * ld(X.mx + q) + wd.y[j] * ld(X.my + q) + wd.z[j] * ld(X.mz + q);
      const Q4<R> av = ld4(av4, (size_t)q);
      sa0 += av.x * f;
      sa1 += av.y * f;
      sa2 += av.z * f;
      if constexpr (SH) sa3 += ld(T.wc + q) * f;
      sdh += f;
      sdt += (SH ? ld(T.theta + q) : av.w) * f;
      const R pq = ld(T.pp + q);
      if constexpr (kByDifference) {
        if (j == 0) {
          p0 = pq;
        } else {
          gx += wd.x[j] * (pq - p0);
          gy += wd.y[j] * (pq - p0);
          gz += wd.z[j] * (pq - p0);
        }
      } else {
        gx += wd.x[j] * pq;
        gy += wd.y[j] * pq;
        gz += wd.z[j] * pq;
        if (j == 0) {
          gx += gcx * pq;
          gy += gcy * pq;
          gz += gcz * pq;
        }
      }
      if (hyper) {
        const Q4<R> hq = ld4(T.q4, (size_t)q);
        hr += wl.v[j] * hq.w;
        hx += wl.v[j] * hq.x;
        hy += wl.v[j] * hq.y;
        hz += wl.v[j] * hq.z;
        hT += wl.v[j] * ld(T.qT + q);
      }
    }

    // hyperdiffusion (Sec. 4)
    R Frho = 0, FMx = 0, FMy = 0, FMz = 0, Fth = 0;
    if (hyper) {
      Frho = -hr * inv_r2;
      FMx = -hx * inv_r2;
      FMy = -hy * inv_r2;
      FMz = -hz * inv_r2;
      Fth = -Rd * hT * inv_r2 / ld(SL.pi + (i));     // Th / (gamma p) F_p
    }

    // advection div(rho v v_j) of the Cartesian components (Sec. 3)
    const R sa[3] = {sa0, sa1, sa2};
    R A[3];
    R wlo_w = ld(X.w + (i)), whi_w = ld(X.w + (i + S));
    // the advected velocity at the cell's lower and upper interfaces
    Q4<R> vl = {0, 0, 0, 0}, vh = {0, 0, 0, 0};
    if constexpr (HO) {
      if (k >= 1) vl = vint_iface4(U, av4, k, c, S, G.nv);
      if (k + 1 < G.nv) vh = vint_iface4(U, av4, k + 1, c, S, G.nv);
    } else {
      const Q4<R> v0 = ld4(av4, (size_t)i);
      if (k >= 1) {
        const Q4<R> vm = ld4(av4, (size_t)(i - S));
        const R a = ld(U.wlo + (k)), b = ld(U.whi + (k));
        vl = {a * vm.x + b * v0.x, a * vm.y + b * v0.y, a * vm.z + b * v0.z, 0};
      }
      if (k + 1 < G.nv) {
        const Q4<R> vp = ld4(av4, (size_t)(i + S));
        const R a = ld(U.wlo + (k + 1)), b = ld(U.whi + (k + 1));
        vh = {a * v0.x + b * vp.x, a * v0.y + b * vp.y, a * v0.z + b * vp.z, 0};
      }
    }
    const R vlo3[3] = {vl.x, vl.y, vl.z}, vhi3[3] = {vh.x, vh.y, vh.z};
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      R ah = sa[j] * inv_r;
      A[j] = ah + sqh * whi_w * vhi3[j] - sql * wlo_w * vlo3[j];
    }
    R acr;
    if constexpr (SH) {
      // traditional Coriolis f r x M_h, f = 2 Omega sin(lat); w advected as a scalar
      const R mx = ld(X.mx + (i)), my = ld(X.my + (i)), mz = ld(X.mz + (i)), f = two_om * rz;
      A[0] += f * (ry * mz - rz * my);
      A[1] += f * (rz * mx - rx * mz);
      A[2] += f * (rx * my - ry * mx);
      R wlo_c = 0, whi_c = 0;
      if constexpr (HO) {
        if (k >= 1) wlo_c = vint_iface(U, (const R*)T.wc, (const R*)nullptr, k, c, S, G.nv);
        if (k + 1 < G.nv) whi_c = vint_iface(U, (const R*)T.wc, (const R*)nullptr, k + 1, c, S, G.nv);
      } else {
        if (k >= 1) wlo_c = ld(U.wlo + (k)) * ld(T.wc + (i - S)) + ld(U.whi + (k)) * ld(T.wc + (i));
        if (k + 1 < G.nv) whi_c = ld(U.wlo + (k + 1)) * ld(T.wc + (i)) + ld(U.whi + (k + 1)) * ld(T.wc + (i + S));
      }
      acr = sa3 * inv_r + sqh * whi_w * whi_c - sql * wlo_w * wlo_c;
    } else {
      // Coriolis 2 Omega z x (rho v) with the full momentum
      R wc = HO ? vint_centre(U, X.w, k, c, S, G.nv) : ld(U.clo + (k)) * wlo_w + ld(U.chi + (k)) * whi_w;
      R mx = ld(X.mx + (i)), my = ld(X.my + (i));
      R fx = mx + wc * rx, fy = my + wc * ry;
      A[0] += -two_om * fy;
      A[1] += two_om * fx;
      acr = A[0] * rx + A[1] * ry + A[2] * rz;
    }

    // the anelastic switch leaves the pressure force to the projection
    const R pgr = ph.anelastic ? R(0) : inv_r;
    // Float: the advection's and the diffusion's radial parts go first, since a
    // radial part leaks into the tangential one by the rounding of the basis
    if constexpr (kByDifference) {
      const R d = SH ? A[0] * rx + A[1] * ry + A[2] * rz : acr, f = FMx * rx + FMy * ry + FMz * rz;
      A[0] -= d * rx;
      A[1] -= d * ry;
      A[2] -= d * rz;
      FMx -= f * rx;
      FMy -= f * ry;
      FMz -= f * rz;
    }
    // the tangential part of the sum, in the basis the small step works in
    // (tan_to with X = s rx, Y = s ry, s = sign(rz): one register instead of three)
    const R sx = -gx * pgr - A[0] + FMx, sy = -gy * pgr - A[1] + FMy, sz = -gz * pgr - A[2] + FMz;
    const R t = tA * (rx * sx + ry * sy) - (rz < R(0) ? -sz : sz);
    st2(SL.sm2, i, sx + rx * t, sy + ry * t);

    R dh = sdh * inv_r;
    R dv = sqh * whi_w - sql * wlo_w;
    SL.srho[i] = -dh - dv + Frho;
    SL.dsc[i] = dh + dv;
    if (d0) d0[i] = dh + dv;

    R dht = sdt * inv_r;
    R thlo = 0, thhi = 0;
    if (k >= 1) thlo = ld(U.wlo + (k)) * ld(T.theta + (i - S)) + ld(U.whi + (k)) * ld(T.theta + (i));
    if (k + 1 < G.nv) thhi = ld(U.wlo + (k + 1)) * ld(T.theta + (i)) + ld(U.whi + (k + 1)) * ld(T.theta + (i + S));
    R dvt = sqh * thhi * whi_w - sql * thlo * wlo_w;
    SL.sth[i] = Fth - dht - dvt;
    SL.acr[i] = acr;
  }
}

// Slow tendency of the vertical momentum at the interior interfaces
// (right-hand side of Eq. momr2) and theta at the interfaces; with init, on
// the same (column, level) grid, also the perturbations at the start of the
// stage: Phi* = Phi^t - Phi^(s), p* from the nonlinear Eq. theta_to_p.
// XtL (init only): the low parts of a compensated X^t (null pointers when X
// is X^t itself or the state is not compensated); the stage state is stored
// as floats
template <typename R, bool HO = false>
__device__ __forceinline__ void d_slow_w(const Geo<R>& G, const VR<R>& U, const Phys& ph, const Xf<R>& Xt, const Xf<R>& X, const Work<R>& T, const Slow<R>& SL,
                                         const Pert<R>& P, int hyper, int init, int kchunk, int bx, int by,
                                         const Xf<R>& XtL = Xf<R>{}) {
  int c = bx * blockDim.x + threadIdx.x;
  pdl_next();
  if (c >= G.ncol) return;
  Nbr7 nb = load_nbr(G, c);
  W7<R> wl = load_w7(G.wlap, G.colp, c);
  const Tan<R> tb = load_tan(G.tb, G.colp, c);
  const int S = pdl_wait(G.colp);
  const R g = pc<R>(ph.g, ph.g_f);
  int k0 = by * kchunk, k1 = min(G.nv + 1, k0 + kchunk);
#pragma unroll 2
  for (int k = k0; k < k1; ++k) {
    const int i = k * S + c;
    // stage start (unless k_stage_init does it)
    auto dif = [&](const R* a, const R* b, const R* al) {
      R d = ld(a + (i)) - ld(b + (i));
      if (al) d += ld(al + (i));
      return d;
    };
    if (init && k < G.nv) {
      P.rho[i] = dif(Xt.rho, X.rho, XtL.rho);
      const Q2<R> m = tan_to(tb, dif(Xt.mx, X.mx, XtL.mx), dif(Xt.my, X.my, XtL.my), dif(Xt.mz, X.mz, XtL.mz));
      st2(P.m2, i, m.x, m.y);
      const R d = dif(Xt.th, X.th, XtL.th);
      P.th[i] = d;
      P.p[i] = p_pert(ph, ld(SL.pi + (i)), ld(U.thb + (k)) + ld(X.th + (i)), d);
    }
    if (init) P.w[i] = dif(Xt.w, X.w, XtL.w);
    // slow terms of Eq. momr2
    if (k == 0 || k == G.nv) {
      SL.sw[i] = 0;
      SL.thi[i] = 0;
      continue;
    }
    R wlo = ld(U.wlo + (k)), whi = ld(U.whi + (k));
    R sw;
    if (ph.anelastic) {
      // Ogura-Phillips buoyancy g rho0_i (theta' / theta0)_i, theta' / theta0 =
      // Th' / Th_bar at rho = rho_bar, both interpolated linearly
      sw = g * (wlo * ld(U.rhob + (k - 1)) + whi * ld(U.rhob + (k)))
           * (wlo * ld(X.th + (i - S)) / ld(U.thb + (k - 1)) + whi * ld(X.th + (i)) / ld(U.thb + (k)));
    } else {
      sw = ld(U.Rb + (k)) - (ld(T.pp + (i)) - ld(T.pp + (i - S))) * ld(U.inv_dzc + (k))
           - g * (wlo * ld(X.rho + (i - S)) + whi * ld(X.rho + (i)));
    }
    // the vertical advection, Coriolis and diffusion of W are part of the
    // inertia that the hydrostatic switch drops
    if (!ph.hydrostatic) {
      R FW = 0;
      if (hyper) FW = div_by(-apply7(wl, nb, T.qvr + k * S), ld(U.ri2 + (k)), ld(U.inv_ri2 + (k)));
      const R acr_i = HO ? vint_iface(U, (const R*)SL.acr, (const R*)nullptr, k, c, S, G.nv)
                                    : wlo * ld(SL.acr + (i - S)) + whi * ld(SL.acr + (i));
      sw = sw - acr_i + FW;
    }
    SL.sw[i] = sw;
    SL.thi[i] = wlo * ld(T.theta + (i - S)) + whi * ld(T.theta + (i));
  }
}

// The perturbations at the start of a stage on their own (the state's step
// runs this beside the slow terms): Phi* = Phi^t - Phi^(s), p* from the
// nonlinear Eq. theta_to_p about the stage state (p_pert); all zero in the
// first stage, where Phi^(s) = Phi^t. M* is tangent (the difference of two states
// with the same radial part) and kept in the column's basis. XtL: the low
// parts of a compensated X^t (null pointers: none), XL those of the stage
// state (null: stored as floats), so that Phi^t - Phi^(s) is taken from the
// full values.
template <typename R>
__device__ __forceinline__ void d_stage_init(const Geo<R>& G, const VR<R>& U, const Phys& ph, const Xf<R>& Xt, const Xf<R>& X, const R* pi, const Pert<R>& P,
                                             const Xf<R>& XtL, const Xf<R>& XL, int zero, int kchunk, int bx, int by) {
  int c = bx * blockDim.x + threadIdx.x;
  pdl_next();
  if (c >= G.ncol) return;
  const Tan<R> tb = load_tan(G.tb, G.colp, c);
  const int S = pdl_wait(G.colp);
  const bool cmp = XtL.rho != nullptr;
  int k0 = by * kchunk, k1 = min(G.nv + 1, k0 + kchunk);
#pragma unroll 2
  for (int k = k0; k < k1; ++k) {
    const int i = k * S + c;
    // Phi^t - Phi^(s) of one field (the stage state of a compensated state
    // is stored as floats, XL null, except in the first stage where it is
    // X^t itself and the perturbations are zero)
    auto dif = [&](const R* a, const R* b, const R* al, const R* bl) {
      R d = ld(a + i) - ld(b + i);
      if (cmp) d += bl ? ld(al + i) - ld(bl + i) : ld(al + i);
      return d;
    };
    if (k < G.nv) {
      if (zero) {
        P.rho[i] = P.th[i] = P.p[i] = R(0);
        st2(P.m2, i, R(0), R(0));
      } else {
        P.rho[i] = dif(Xt.rho, X.rho, XtL.rho, XL.rho);
        const Q2<R> m = tan_to(tb, dif(Xt.mx, X.mx, XtL.mx, XL.mx), dif(Xt.my, X.my, XtL.my, XL.my),
                               dif(Xt.mz, X.mz, XtL.mz, XL.mz));
        st2(P.m2, i, m.x, m.y);
        const R d = dif(Xt.th, X.th, XtL.th, XL.th);
        P.th[i] = d;
        P.p[i] = p_pert(ph, ld(pi + (i)), ld(U.thb + (k)) + ld(X.th + (i)), d);
      }
    }
    P.w[i] = zero ? R(0) : dif(Xt.w, X.w, XtL.w, XL.w);
  }
}

// ---------------------------------------------------------------- small step

// L2 eviction priorities of the small step's planes (thor_tune
// THOR_TUNE_L2_HINTS): bit 0 loads the stage constants evict-first, bit 1
// keeps the perturbations and the split's intermediates evict-last. Default
// 3 (both): at glevel 6 x 32 levels the large step takes 1.187 ms, against
// 1.192 with the constants' hint alone, 1.227 with the other's and 1.233 without
// hints. Float64 states keep their perturbations at the normal priority whatever
// the mode: their set is twice the size, and held evict-last it slowed the
// float64 large step by an eighth (then 9.85 ms; 6.15 now, in every mode).
__constant__ int c_l2mode = 3;
__device__ __forceinline__ uint64_t pol_stream() { return l2_policy((c_l2mode & 1) ? kL2First : kL2Normal); }
template <typename R = float>
__device__ __forceinline__ uint64_t pol_keep() {
  return l2_policy(sizeof(R) == sizeof(float) && (c_l2mode & 2) ? kL2Last : kL2Normal);
}
int set_l2_mode(int mode) { return cudaMemcpyToSymbol(c_l2mode, &mode, sizeof mode) == cudaSuccess ? 0 : -1; }

template <typename R>
// Divergence damping, first stencil (Sec. 4, reading R5: the damping is
// -K_d grad_h(lap D)): the Laplacian of the 3-D divergence D of the total
// momentum, D = d0 in the first small step of a stage and later the D the
// previous column step formed. The pressure gradient and the damping go
// through the same gradient weights, so what is stored is the one scalar
// q = p* + K_d lap D whose gradient the momentum step takes: one word per
// cell written here and gathered there instead of two, and 21 multiply-adds
// per cell less there. This kernel is bound by its loads' latency; at g6 x 32
// float 11.7 -> 11.6 us, float64 25.4 -> 28.2 us.
__device__ __forceinline__ void d_ss_lapd(const Geo<R>& G, const VR<R>& U, const Work<R>& T, const R* dsrc, const R* pstar, R Kd,
                                          int kchunk, int bx, int by) {
  int c = bx * blockDim.x + threadIdx.x;
  pdl_next();
  if (c >= G.ncol) return;
  const uint64_t pk = pol_keep<R>();
  Nbr7 nb = load_nbr(G, c);
  W7<R> wl = load_w7(G.wlap, G.colp, c);
  const int S = pdl_wait(G.colp);
  int k0 = by * kchunk, k1 = min(G.nv, k0 + kchunk);
#pragma unroll 2
  for (int k = k0; k < k1; ++k) {
    const int o = k * S, i = o + c;
    R l = 0;
#pragma unroll
    for (int j = 0; j < 7; ++j) l += wl.v[j] * ldh(dsrc + (o + nb.n[j]), pk);
    sth(T.lp + i, fmar<R>(l * ld(U.inv_rc2 + (k)), Kd, ldh(pstar + (i), pk)), pk);
  }
}

// Eq. mom2 with the divergence damping: M* <- M* + dtau(-grad q + S_M), in the
// column's tangent basis (so Eq. proj_h is built into the weights),
// q = p* + K_d lap D of d_ss_lapd, or p* itself without the damping; float
// states take the gradient of q less its mean over the seven points (a
// constant has no gradient): the one word q rounds away low bits of its smaller term,
// and the sums of weight times value round on the scale of the values, which
// is many times that of their differences (a long wave at glevel 4: 2.1e-7 of
// the gradient; two stored words 1.7e-7; less the mean 1.1e-7). The 14 operations
// a cell wait for all seven values: g6 x 32 0.4% of a large step, g5 states 0.4 to 2%;
// in the last small step of a stage also M^(s+1) = M^(s) + M* into Xo (which
// may be Xs itself: each cell reads its own Xs value before writing it), with
// the low parts XsL -> XoL of a compensated state (null: none). Bound by the
// gathers' latency (float) and by the float64 pipe's multiply-adds (float64):
// at g6 x 32, float 28.7 us with two gathered scalars and three Cartesian
// components, 25.2 with one scalar, 17.9 in the tangent basis (80 -> 48
// registers); float64 147 -> 84 -> 52 us.
template <typename R>
__device__ __forceinline__ void d_ss_mom(const Geo<R>& G, const VR<R>& U, const Slow<R>& SL, const Pert<R>& P, const Work<R>& T, R dtau,
                                            int divdamp, const Xf<R>& Xs, const Xf<R>& Xo, const Xf<R>& XsL, const Xf<R>& XoL, int last,
                                            int kchunk, int bx, int by) {
  int c = bx * blockDim.x + threadIdx.x;
  pdl_next();
  if (c >= G.ncol) return;
  const uint64_t ps = pol_stream(), pk = pol_keep<R>();
  Nbr7 nb = load_nbr(G, c);
  W7x2<R> wg = load_w7x2(G.wg2, G.colp, c);
  const int S = pdl_wait(G.colp);
  const R* q = divdamp ? T.lp : P.p;
  int k0 = by * kchunk, k1 = min(G.nv, k0 + kchunk);
#pragma unroll 2
  for (int k = k0; k < k1; ++k) {
    const int o = k * S, i = o + c;
    R inv_r = ld(U.inv_rc + (k));
    R v[7], g1 = 0, g2 = 0;
#pragma unroll
    for (int j = 0; j < 7; ++j) v[j] = ldh(q + (o + nb.n[j]), pk);
    if constexpr (sizeof(R) == sizeof(float)) {
      const R sum = ((v[1] + v[2]) + (v[3] + v[4])) + ((v[5] + v[6]) + v[0]);
#pragma unroll
      for (int j = 0; j < 7; ++j) v[j] = fmar<R>(sum, R(-1.0 / 7.0), v[j]);
    }
#pragma unroll
    for (int j = 0; j < 7; ++j) {
      g1 += wg.x[j] * v[j];
      g2 += wg.y[j] * v[j];
    }
    Q2<R> m = ld2h(P.m2, (size_t)i, pk);
    const Q2<R> sm = ld2h(SL.sm2, (size_t)i, ps);
    m.x += dtau * fmar<R>(-g1, inv_r, sm.x);
    m.y += dtau * fmar<R>(-g2, inv_r, sm.y);
    st2h(P.m2, i, m.x, m.y, pk);
    if (last) {          // end of the stage: M^(s+1) = M^(s) + M*
      R mx, my, mz;
      tan_from(load_tan(G.tb, S, c), m, mx, my, mz);
      if (XoL.mx) {
        comp_add<R>(Xs.mx, XsL.mx, Xo.mx, XoL.mx, i, mx);
        comp_add<R>(Xs.my, XsL.my, Xo.my, XoL.my, i, my);
        comp_add<R>(Xs.mz, XsL.mz, Xo.mz, XoL.mz, i, mz);
      } else {
        Xo.mx[i] = ld(Xs.mx + (i)) + mx;
        Xo.my[i] = ld(Xs.my + (i)) + my;
        Xo.mz[i] = ld(Xs.mz + (i)) + mz;
      }
    }
  }
}

// HE-VI column step, part 1: horizontal fluxes of the new M* and, for every
// cell, the parts of Eqs. dens2 and pt2 that do not involve W*:
//   a_k = rho*_k + dtau (S_rho,k - div_h M*_k)
//   b_k = Th*_k + dtau (S_th,k - div_h(theta M*)_k)
//   c_k = p*_k + Pi_k (b_k - Th*_k)        (p* advanced linearly in Th)
// M* comes in the tangent basis of each neighbour (two multiply-adds per edge
// instead of three); at g6 x 32 float64 107 -> 90 us (float64 pipe), float
// 22.5 -> 22.9 us (latency: the gather of theta beside M* is its own load now)
template <typename R>
struct FluxCell {
  R dhm, a, b, c;
};
// the four values of cell i = o + column (o = level k's plane offset)
template <typename R>
__device__ __forceinline__ FluxCell<R> flux_cell(const W7x2<R>& wd, const Nbr7& nb, const VR<R>& U,
                                                 const Slow<R>& SL, const Pert<R>& P, const Work<R>& T, R dtau,
                                                 int k, int o, int i, uint64_t ps, uint64_t pk) {
  R dh = 0, dht = 0;
#pragma unroll
  for (int j = 0; j < 7; ++j) {
    const Q2<R> m = ld2h(P.m2, (size_t)(o + nb.n[j]), pk);    // M* of the neighbour in its basis
    const R f = fmar<R>(wd.y[j], m.y, wd.x[j] * m.x);
    dh += f;
    dht += ldh(T.theta + (o + nb.n[j]), pk) * f;
  }
  const R inv_r = ld(U.inv_rc + (k));
  const R thk = ldh(P.th + (i), pk);
  const R bk = thk + dtau * (ldh(SL.sth + (i), ps) - dht * inv_r);
  FluxCell<R> r;
  r.dhm = dh * inv_r;
  r.a = ldh(P.rho + (i), pk) + dtau * (ldh(SL.srho + (i), ps) - dh * inv_r);
  r.b = bk;
  r.c = ldh(P.p + (i), pk) + ldh(SL.pi + (i), ps) * (bk - thk);
  return r;
}

template <typename R>
__device__ __forceinline__ void d_ss_flux(const Geo<R>& G, const VR<R>& U, const Slow<R>& SL, const Pert<R>& P, const Work<R>& T, R dtau, int kchunk, int bx, int by) {
  int c = bx * blockDim.x + threadIdx.x;
  pdl_next();
  if (c >= G.ncol) return;
  const uint64_t ps = pol_stream(), pk = pol_keep<R>();
  Nbr7 nb = load_nbr(G, c);
  W7x2<R> wd = load_w7x2(G.wd2, G.colp, c);
  const int S = pdl_wait(G.colp);
  int k0 = by * kchunk, k1 = min(G.nv, k0 + kchunk);
#pragma unroll 2
  for (int k = k0; k < k1; ++k) {
    const int o = k * S, i = o + c;
    const FluxCell<R> f = flux_cell(wd, nb, U, SL, P, T, dtau, k, o, i, ps, pk);
    sth(T.dhm + i, f.dhm, pk);
    sth(T.ca + i, f.a, pk);
    sth(T.cb + i, f.b, pk);
    sth(T.cc + i, f.c, pk);
  }
}

// one row's factors of a float64 state
template <typename R>
__device__ __forceinline__ void fac_store(const Fac<R>& F, int i, double inv, double cf, double q) {
  F.inv[i] = inv;
  F.cf[i] = cf;
  F.q[i] = q;
}

// HE-VI column step, part 2 (matrix). Substituting Eqs. dens2 and pt2 into
// Eq. momr2 gives at the interior interfaces m = 1..nv-1 (rigid lid: W* = 0
// at m = 0 and nv)
//   lo_m W_m-1 + di_m W_m + up_m W_m+1 = rh_m
// with e_k = r^2/(rc_k^2 dz_k) at the bottom (sq_lo) and top (sq_hi)
// interfaces of cell k, th_m = theta at interface m, w-/w+ the Lagrange
// weights of centres m-1, m at interface m:
//   lo_m = -dtau^2/dzc_m Pi_m-1 sq_lo_m-1 th_m-1 + dtau^2 g w- sq_lo_m-1
//   di_m = 1 + dtau^2/dzc_m th_m (Pi_m sq_lo_m + Pi_m-1 sq_hi_m-1)
//            - dtau^2 g (w- sq_hi_m-1 - w+ sq_lo_m)
//   up_m = -dtau^2/dzc_m Pi_m sq_hi_m th_m+1 - dtau^2 g w+ sq_hi_m
// The matrix depends only on the stage state (Pi, theta) and dtau, so it is
// factorised once per RK stage and the factors serve every small step of
// the stage. The factorisation is the matrix half of a two-sided Thomas
// algorithm, in float64 for float64 states and in double-float (df_rcp,
// df_mul_f: pivot reciprocals to about 2^-46) for float-storage states:
// one half of the lanes eliminates rows 1..p downwards
// (c'_m = up_m / (di_m - lo_m c'_m-1)), the other rows nv-1..p+1 upwards
// (e'_m = lo_m / (di_m - up_m e'_m+1)). Stored per row (Fac): the pivot
// reciprocal, and in float64 c' or e' and q = lo or up times the reciprocal, in
// float storage lo and up themselves; per column: 1 / (1 - c'_p e'_p+1) for the
// junction rows p, p+1.
//
// the matrix row m of column c in the storage type
template <typename R>
__device__ __forceinline__ void matrix_row(const VR<R>& U, const Slow<R>& SL, R g, R dt2, R delta, int nv, int S, int c,
                                           int m, R& lo, R& di, R& up) {
  const int i = m * S + c, N = nv - 1;
  const R pi_lo = ld(SL.pi + (i - S)), pi_hi = ld(SL.pi + i);
  const R wlo = ld(U.wlo + m), whi = ld(U.whi + m), dtz = dt2 * ld(U.inv_dzc + m);
  const R ql = ld(U.sq_lo + (m - 1)), qh = ld(U.sq_hi + (m - 1));   // cell m-1
  const R pl = ld(U.sq_lo + m), ph_ = ld(U.sq_hi + m);              // cell m
  const R th_m = ld(SL.thi + i);
  R lower = 0, upper = 0;
  if (m > 1) lower = (-dtz * pi_lo * ld(SL.thi + (i - S)) + dt2 * g * wlo) * ql;
  if (m < N) upper = (-dtz * pi_hi * ld(SL.thi + (i + S)) - dt2 * g * whi) * ph_;
  lo = lower;
  up = upper;
  di = delta + dtz * th_m * (pi_hi * pl + pi_lo * qh) - dt2 * g * (wlo * qh - whi * pl);
}

// float storage: 32 columns a block, one warp for each of the two sweeps
__device__ __forceinline__ void d_ss_factor(const Geo<float>& G, const VR<float>& U, const Phys& ph,
                                            const Slow<float>& SL, const Fac<float>& F, double dtau, int bx) {
  pdl_next();
  const int nv = G.nv, S = pdl_wait(G.colp), N = nv - 1;
  const int tx = threadIdx.x & 31, half = threadIdx.x >> 5;
  const int c = bx * 32 + tx;
  const bool valid = c < G.ncol;
  const int cs = valid ? c : 0;          // padding lanes compute on column 0 and store nothing
  const int p = N / 2 > 0 ? N / 2 : 1;
  const float g = ph.g_f, dt2 = (float)(dtau * dtau), delta = ph.delta_f;
  auto coef_r = [&](int m, float& lo, float& di, float& up) {
    matrix_row<float>(U, SL, g, dt2, delta, nv, S, cs, m, lo, di, up);
  };
  // float storage: the factorisation in double-float on the float32 pipes
  // (the float coefficients are exact pairs), stored as pairs
  __shared__ float2 sj2[2][32];
  float2* Finv = reinterpret_cast<float2*>(F.inv);
  float* Flo = reinterpret_cast<float*>(F.q);
  float* Fup = reinterpret_cast<float*>(F.cf);
  float2 last = make_float2(0.f, 0.f);
  if (half == 0) {
    for (int m = 1; m <= p; ++m) {
      float lo, di, up;
      coef_r(m, lo, di, up);
      const float2 inv = df_rcp(df_fms(di, 0.f, make_float2(lo, 0.f), last));
      last = df_mul_f(up, inv);
      if (valid) {
        Finv[m * S + c] = inv;
        Flo[m * S + c] = lo;
        Fup[m * S + c] = up;
      }
    }
  } else {
    for (int m = N; m > p; --m) {
      float lo, di, up;
      coef_r(m, lo, di, up);
      const float2 inv = df_rcp(df_fms(di, 0.f, make_float2(up, 0.f), last));
      last = df_mul_f(lo, inv);
      if (valid) {
        Finv[m * S + c] = inv;
        Flo[m * S + c] = lo;
        Fup[m * S + c] = up;
      }
    }
  }
  sj2[half][tx] = last;    // c'_p (warp 0) and e'_p+1 (warp 1)
  __syncthreads();
  if (half == 0 && valid)
    reinterpret_cast<float2*>(F.junction)[c] =
        p < N ? df_rcp(df_fms(1.f, 0.f, sj2[0][tx], sj2[1][tx])) : make_float2(1.f, 0.f);
}

// Float64 columns: a block is kCols64 = 16 columns x 16 threads each. The
// matrix rows (and the solve's right-hand sides and final updates) are shared
// by all sixteen; lanes 0-15 of one warp then run the downward sweep and lanes
// 16-31 the upward one, in the same instructions, each over shared memory.
// A float64 warp instruction holds its sub-partition's pipe for 80 cycles, so
// what a small grid needs is every SM: 16 columns a block give a g4 grid 161
// blocks for 152 SMs where 32 gave it 81. The large step against 32 columns a
// block: g4 x 20 430 -> 411 us, g5 x 32 1577 -> 1507 us, g6 x 32 6085 -> 6132
// us (there every SM is busy either way). With 64 / 128 / 256 threads a block
// in both kernels: g4 508 / 438 / 418, g5 1651 / 1554 / 1508, g6 6108 / 6113 /
// 6142 us.
constexpr int kCols64 = 16, kThreads64 = 256;
struct Lane64 {
  int tx, slot, c, cs;
  bool valid, sweeps;
  __device__ Lane64(int bx, int ncol) {
    tx = threadIdx.x & (kCols64 - 1);
    slot = threadIdx.x / kCols64;
    c = bx * kCols64 + tx;
    valid = c < ncol;
    cs = valid ? c : 0;                  // padding lanes compute on column 0 and store nothing
    // the sweeping warp differs from block to block, so that the blocks of an
    // SM do not all sweep on one sub-partition
    sweeps = (threadIdx.x >> 5) == ((unsigned)bx * 2654435761u >> 29);
  }
};

__device__ __forceinline__ void d_ss_factor(const Geo<double>& G, const VR<double>& U, const Phys& ph,
                                            const Slow<double>& SL, const Fac<double>& F, double dtau, int bx) {
  extern __shared__ double sm[];
  pdl_next();
  const int nv = G.nv, S = pdl_wait(G.colp), N = nv - 1;
  const Lane64 L(bx, G.ncol);
  const int p = N / 2 > 0 ? N / 2 : 1, rows = (nv + 1) * kCols64;
  double *slo = sm, *sdi = sm + rows, *sup = sm + 2 * rows;      // [nv + 1][kCols64] each
  for (int m = 1 + L.slot; m <= N; m += kThreads64 / kCols64) {
    const int o = m * kCols64 + L.tx;
    matrix_row<double>(U, SL, ph.g, dtau * dtau, ph.delta, nv, S, L.cs, m, slo[o], sdi[o], sup[o]);
  }
  __syncthreads();
  if (!L.sweeps) return;
  const bool down = (L.slot & 1) == 0;
  const int len = down ? p : N - p;
  const double *off = down ? slo : sup, *oth = down ? sup : slo;
  double last = 0.0;
  for (int t = 0; t < len; ++t) {
    const int m = down ? 1 + t : N - t, o = m * kCols64 + L.tx;
    const double a = off[o], inv = 1.0 / (sdi[o] - a * last);
    last = oth[o] * inv;
    if (L.valid) fac_store(F, m * S + L.c, inv, last, a * inv);
  }
  __syncwarp();
  const double e = __shfl_down_sync(0xffffffffu, last, kCols64);     // e'_p+1 beside c'_p
  if (down && L.valid) F.junction[L.c] = p < N ? 1.0 / (1.0 - last * e) : 1.0;
}

// End of an RK stage for one cell of the column step: Phi^(s+1) = Phi^(s) +
// Phi* for rho, rho theta and W (the momentum in k_ss_mom), into Xo, which may
// be Xs itself (each cell reads its own Xs values before writing them). The
// lid and surface interfaces keep W^(s) + W*, as the interior ones.
// XsL, XoL: the low parts of a compensated state (null: none), updated
// with comp_add so that the stage end does not round the state.
template <typename R>
__device__ __forceinline__ void stage_end_cell(const Xf<R>& Xs, const Xf<R>& Xo, const Xf<R>& XsL, const Xf<R>& XoL,
                                               const Pert<R>& P, R rho_new, R th_new, R w_new, int k, int i, int S,
                                               int nv) {
  if (XoL.rho) {
    comp_add<R>(Xs.rho, XsL.rho, Xo.rho, XoL.rho, i, rho_new);
    comp_add<R>(Xs.th, XsL.th, Xo.th, XoL.th, i, th_new);
    if (k >= 1) comp_add<R>(Xs.w, XsL.w, Xo.w, XoL.w, i, w_new);
    if (k == 0) comp_add<R>(Xs.w, XsL.w, Xo.w, XoL.w, i, ld(P.w + i));
    if (k == nv - 1) comp_add<R>(Xs.w, XsL.w, Xo.w, XoL.w, i + S, ld(P.w + (i + S)));
    return;
  }
  Xo.rho[i] = ld(Xs.rho + i) + rho_new;
  Xo.th[i] = ld(Xs.th + i) + th_new;
  if (k >= 1) Xo.w[i] = ld(Xs.w + i) + w_new;
  if (k == 0) Xo.w[i] = ld(Xs.w + i) + ld(P.w + i);
  if (k == nv - 1) Xo.w[i + S] = ld(Xs.w + (i + S)) + ld(P.w + (i + S));
}

constexpr int kSolveWarps = 8;     // warps of a column solve's block

// HE-VI column step, part 3 (every small step). The right-hand side
//   rh_m = W*_m + dtau S_W,m - dtau/dzc_m (c_m - c_m-1) - dtau g (w- a_m-1 + w+ a_m)
// goes through the stored factors (d'_m = rh_m / piv_m - q_m d'_m-1
// downwards, f'_m = rh_m / piv_m - q_m f'_m+1 upwards: one dependent
// multiply-add per row, the product rh_m / piv_m off the chain; then the
// junction rows x_p = (d'_p - c'_p f'_p+1) / (1 - c'_p e'_p+1),
// x_p+1 = f'_p+1 - e'_p+1 x_p, then back substitution outwards), in float64
// for float64 states and in double-float for float-storage states; then
// rho* and Th* follow from Eqs. dens2 and pt2 and p* from the nonlinear Eq.
// theta_to_p.
//
// The cell's update with the solved W* at its interfaces (wl, wh):
template <typename R>
__device__ __forceinline__ void update_cell(const VR<R>& U, const Phys& ph, const Xf<R>& Xs, const Slow<R>& SL,
                                            const Pert<R>& P, const Work<R>& T, R rdt, R wl, R wh, int want_div,
                                            const Xf<R>& Xo, const Xf<R>& XsL, const Xf<R>& XoL, int last, int k, int i,
                                            int S, int nv) {
  const R thl = k > 0 ? ld(SL.thi + i) : R(0);
  const R thh = k + 1 < nv ? ld(SL.thi + (i + S)) : R(0);
  const R el = ld(U.sq_lo + k), eh = ld(U.sq_hi + k);
  R th_new = ld(T.cb + i) - rdt * (eh * thh * wh - el * thl * wl);
  const R rho_new = ld(T.ca + i) - rdt * (eh * wh - el * wl);
  P.rho[i] = rho_new;
  P.th[i] = th_new;
  // p* = EOS(Th^(s) + Th*) - p^(s)
  P.p[i] = p_pert(ph, ld(SL.pi + i), ld(U.thb + k) + ld(Xs.th + i), th_new);
  if (k >= 1) P.w[i] = wl;
  // 3-D divergence of the new total momentum, for the next small step's
  // divergence damping: D^(s) + div_h M* (from k_ss_flux) + div_v W*
  if (want_div) T.dd[i] = ld(SL.dsc + i) + ld(T.dhm + i) + (eh * wh - el * wl);
  if (last) stage_end_cell(Xs, Xo, XsL, XoL, P, rho_new, th_new, wl, k, i, S, nv);
}

// One block = 32 columns x 8 warps, float storage where the staged solve does
// not apply: two warps sweep, all share the levels of the final updates.
__device__ __forceinline__ void d_ss_solve(const Geo<float>& G, const VR<float>& U, const Phys& ph, const Xf<float>& Xs,
                                            const Slow<float>& SL, const Pert<float>& P, const Work<float>& T,
                                            const Fac<float>& F, double dtau, int want_div, const Xf<float>& Xo,
                                            const Xf<float>& XsL, const Xf<float>& XoL, int last, int bx) {
  using R = float;
  extern __shared__ double sm[];
  pdl_next();
  const int nv = G.nv, S = pdl_wait(G.colp), N = nv - 1;
  const int tx = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int c = pdl_wait(bx * 32 + tx);
  const bool valid = c < G.ncol;
  const int cs = valid ? c : 0;          // padding lanes read column 0 and store nothing
  double* sdp = sm;                      // [nv + 1][32] d' / f', then W
  double* sx = sdp + (nv + 1) * 32;      // [2][32] junction values
  double* scf = sx + 64;                 // [nv + 1][32] c' / e', fetched during the sweeps
  const int p = N / 2 > 0 ? N / 2 : 1;
  const R rdt = (R)dtau, g = pc<R>(ph.g, ph.g_f), delta = pc<R>(ph.delta, ph.delta_f);

  auto rhs_r = [&](int m) {
    const int i = m * S + cs;
    const R wlo = ld(U.wlo + m), whi = ld(U.whi + m);
    return delta * ld(P.w + i) + rdt * ld(SL.sw + i) - rdt * ld(U.inv_dzc + m) * (ld(T.cc + i) - ld(T.cc + (i - S)))
           - rdt * g * (wlo * ld(T.ca + (i - S)) + whi * ld(T.ca + i));
  };
  // float storage: the elimination in double-float, the same operations
  // in the same order as the staged solve (solve_sweeps); W* (float) over
  // the first word of each row of sdp
  const float* Flo = reinterpret_cast<const float*>(F.q);
  const float2* Finv = reinterpret_cast<const float2*>(F.inv);
  const float* Fup = reinterpret_cast<const float*>(F.cf);
  float2* dp2 = reinterpret_cast<float2*>(sdp);
  float2* sx2 = reinterpret_cast<float2*>(sx);
  float2* cf2 = reinterpret_cast<float2*>(scf);
  if (warp == 0) {
    float2 d1 = make_float2(0.f, 0.f);
#pragma unroll 4
    for (int m = 1; m <= p; ++m) {
      const int i = m * S + cs;
      const float2 inv = Finv[i];
      cf2[m * 32 + tx] = df_mul_f(Fup[i], inv);
      d1 = df_sweep(rhs_r(m), inv, df_mul_f(Flo[i], inv), d1);
      dp2[m * 32 + tx] = d1;
    }
  } else if (warp == 1) {
    float2 f1 = make_float2(0.f, 0.f);
#pragma unroll 4
    for (int m = N; m > p; --m) {
      const int i = m * S + cs;
      const float2 inv = Finv[i];
      cf2[m * 32 + tx] = df_mul_f(Flo[i], inv);
      f1 = df_sweep(rhs_r(m), inv, df_mul_f(Fup[i], inv), f1);
      dp2[m * 32 + tx] = f1;
    }
  }
  __syncthreads();
  if (warp == 0) {
    float2 xp, xq = make_float2(0.f, 0.f);
    if (p < N) {
      const float2 dp_ = dp2[p * 32 + tx], fq = dp2[(p + 1) * 32 + tx];
      xp = df_mul(df_fms(dp_.x, dp_.y, cf2[p * 32 + tx], fq), reinterpret_cast<const float2*>(F.junction)[cs]);
      xq = df_fms(fq.x, fq.y, cf2[(p + 1) * 32 + tx], xp);
    } else {
      xp = dp2[p * 32 + tx];
    }
    sx2[tx] = xp;
    sx2[32 + tx] = xq;
  }
  __syncthreads();
  if (warp == 0) {
    float2 x = sx2[tx];
    dp2[p * 32 + tx] = make_float2(df_to_float(x), 0.f);
    for (int m = p - 1; m >= 1; --m) {
      const float2 d = dp2[m * 32 + tx];
      x = df_fms(d.x, d.y, cf2[m * 32 + tx], x);
      dp2[m * 32 + tx] = make_float2(df_to_float(x), 0.f);
    }
    dp2[tx] = make_float2(0.f, 0.f);             // bottom interface
  } else if (warp == 1) {
    float2 x = sx2[32 + tx];
    if (p < N) dp2[(p + 1) * 32 + tx] = make_float2(df_to_float(x), 0.f);
    for (int m = p + 2; m <= N; ++m) {
      const float2 d = dp2[m * 32 + tx];
      x = df_fms(d.x, d.y, cf2[m * 32 + tx], x);
      dp2[m * 32 + tx] = make_float2(df_to_float(x), 0.f);
    }
    dp2[nv * 32 + tx] = make_float2(0.f, 0.f);    // top interface
  }
  __syncthreads();
  // Eqs. dens2, pt2, theta_to_p with the new W*; the warps share the levels
  if (valid) {
#pragma unroll 4
    for (int k = warp; k < nv; k += kSolveWarps) {
      const int i = k * S + c;
      const R wl = dp2[k * 32 + tx].x, wh = dp2[(k + 1) * 32 + tx].x;
      update_cell<R>(U, ph, Xs, SL, P, T, rdt, wl, wh, want_div, Xo, XsL, XoL, last, k, i, S, nv);
    }
  }
}

// Float64 storage (the layout of threads as in the float64 factorisation):
// rh_m / piv_m by all threads, the sweeps and the back substitution one
// multiply-add per row in one warp, the updates by all threads.
__device__ __forceinline__ void d_ss_solve(const Geo<double>& G, const VR<double>& U, const Phys& ph,
                                            const Xf<double>& Xs, const Slow<double>& SL, const Pert<double>& P,
                                            const Work<double>& T, const Fac<double>& F, double dtau, int want_div,
                                            const Xf<double>& Xo, const Xf<double>& XsL, const Xf<double>& XoL, int last,
                                            int bx) {
  extern __shared__ double sm[];
  pdl_next();
  const int nv = G.nv, S = pdl_wait(G.colp), N = nv - 1;
  const Lane64 L(pdl_wait(bx), G.ncol);
  const int p = N / 2 > 0 ? N / 2 : 1, rows = (nv + 1) * kCols64;
  double *sd = sm, *sq = sm + rows;      // [nv + 1][kCols64]: rh / piv, then d' / f', then W; q, then c' / e'
  const double g = ph.g, delta = ph.delta;
  for (int m = 1 + L.slot; m <= N; m += kThreads64 / kCols64) {
    const int i = m * S + L.cs, o = m * kCols64 + L.tx;
    const double rh = delta * ld(P.w + i) + dtau * ld(SL.sw + i)
                      - dtau * ld(U.inv_dzc + m) * (ld(T.cc + i) - ld(T.cc + (i - S)))
                      - dtau * g * (ld(U.wlo + m) * ld(T.ca + (i - S)) + ld(U.whi + m) * ld(T.ca + i));
    sd[o] = rh * ld(F.inv + i);
    sq[o] = ld(F.q + i);
  }
  __syncthreads();
  if (L.sweeps) {
    const bool down = (L.slot & 1) == 0;
    const int len = down ? p : N - p;
    double d = 0.0;
#pragma unroll 4
    for (int t = 0; t < len; ++t) {
      const int m = down ? 1 + t : N - t, o = m * kCols64 + L.tx;
      d = fma(-sq[o], d, sd[o]);
      sd[o] = d;
      sq[o] = ld(F.cf + (m * S + L.cs));
    }
    __syncwarp();
    const int op = p * kCols64 + L.tx, oq = op + kCols64;
    double x = sd[op];
    if (p < N) {
      // x_p, x_p+1
      x = (x - sq[op] * sd[oq]) * ld(F.junction + L.cs);
      if (!down) x = sd[oq] - sq[oq] * x;
    }
    __syncwarp();
    if (down)
      sd[op] = x;
    else if (p < N)
      sd[oq] = x;
    const int back = down ? p - 1 : N - p - 1;
    for (int t = 0; t < back; ++t) {
      const int m = down ? p - 1 - t : p + 2 + t, o = m * kCols64 + L.tx;
      x = sd[o] - sq[o] * x;
      sd[o] = x;
    }
    sd[(down ? 0 : nv) * kCols64 + L.tx] = 0.0;       // bottom and top interfaces
  }
  __syncthreads();
  if (!L.valid) return;
#pragma unroll 2
  for (int k = L.slot; k < nv; k += kThreads64 / kCols64)
    update_cell<double>(U, ph, Xs, SL, P, T, dtau, sd[k * kCols64 + L.tx], sd[(k + 1) * kCols64 + L.tx], want_div, Xo,
                        XsL, XoL, last, k, k * S + L.c, S, nv);
}

// ---------------------------------------------------------------- physics

// Sec. 5 backward-Euler friction (Eq. im_eq_v) and Newtonian relaxation
// (Eq. im_eq_t) with the Sec. 6.1 Held-Suarez or Sec. 6.2 hot-Jupiter
// coefficients; sigma = p / p_s with p_s extrapolated hydrostatically at the
// lowest layer's temperature.
// p_s (and 1 / p_s, div_by) of every column before the physics update, from its lowest layer
// (one thread per column; the update kernel then works on chunks of levels
// and changes the lowest layer's rho theta)
template <typename R>
__device__ __forceinline__ void d_surface_p(const Geo<R>& G, const VR<R>& U, const Phys& ph, const Xf<R>& X, const Work<R>& T, int bx) {
  pdl_next();
  const int c = pdl_wait((int)(bx * blockDim.x + threadIdx.x));
  if (c >= G.ncol) return;
  const R Rd = pc<R>(ph.Rd, ph.Rd_f);
  R p0 = ld(U.pb + (0)) + eos_level(U, ph, 0, ld(X.th + (c)));
  R T0 = p0 / ((ld(U.rhob + (0)) + ld(X.rho + (c))) * Rd);
  const R ps = p0 * rexp<R>(pc<R>(ph.g, ph.g_f) * ld(U.zc + (0)) / (Rd * T0));
  T.psurf[c] = ps;
  T.psurf[G.colp + c] = R(1) / ps;
}

// XL: the low parts of a compensated state (null: none); there the friction
// and the relaxation enter as increments of the state's pairs, the same
// update written as M (1/(1 + K_v dt) - 1) and rho theta at fixed rho
// scaled by (T_new / T)^(1/gamma).
template <typename R>
__device__ __forceinline__ void d_physics(const Geo<R>& G, const VR<R>& U, const Phys& ph, const Xf<R>& X, const Xf<R>& XL, const Work<R>& T, int forcing,
                                          double dt, double hj_dT, int kchunk, int bx, int by) {
  pdl_next();
  const int c = pdl_wait((int)(bx * blockDim.x + threadIdx.x));
  if (c >= G.ncol) return;
  const int S = G.colp;
  const R gamma = pc<R>(ph.gamma, ph.gamma_f), inv_gamma = pc<R>(ph.inv_gamma, ph.inv_gamma_f),
          Rd = pc<R>(ph.Rd, ph.Rd_f), kappa = pc<R>(ph.kappa, ph.kappa_f);
  R sl = ld(G.sinlat + (c)), cl = ld(G.coslat + (c)), clcl = ld(G.xdir + (c));
  const R ps = ld(T.psurf + (c)), inv_ps = ld(T.psurf + (S + c));
  const R rdt = (R)dt;
  const int k0 = by * kchunk, k1 = min(G.nv, k0 + kchunk);
  const bool cmp = XL.rho != nullptr;
  for (int k = k0; k < k1; ++k) {
    const int i = k * S + c;
    R rhop = cmp ? ld(X.rho + (i)) + ld(XL.rho + (i)) : ld(X.rho + (i));
    const R thp = cmp ? ld(X.th + (i)) + ld(XL.th + (i)) : ld(X.th + (i));
    R rho = ld(U.rhob + (k)) + rhop;
    // p and, for Held-Suarez, ln(p / p0) and (p / p0)^kappa, kappa gamma =
    // gamma - 1; float64 takes all three from one table row
    const R p00 = R(1.0e5);
    R p, lpr = 0, prk = 0;
    if constexpr (sizeof(R) == sizeof(double)) {
      const double x = div_by(thp, ld(U.thb + (k)), ld(U.inv_thb + (k)));
      double f, l;
      if (!pow1p<true>(ph, U.pw, x, f, l)) {
        const double2 g = pow1p_general(x, gamma);
        f = g.x;
        l = g.y;
      }
      p = ld(U.pb + (k)) * (1.0 + f);
      if (forcing == THOR_FORCING_HELD_SUAREZ) {
        lpr = fma(gamma, l, ld(U.lnp0 + (k)));
        prk = ld(U.pk0 + (k)) * (1.0 + f) / (1.0 + x);
      }
    } else {
      p = ld(U.pb + (k)) + eos_level(U, ph, k, thp);
      if (forcing == THOR_FORCING_HELD_SUAREZ) {
        lpr = rlog<R>(p / p00);
        prk = rpow<R>(p / p00, kappa);
      }
    }
    R Temp = p / (rho * Rd);
    R sigma = div_by(p, ps, inv_ps);
    R Kv, KT, Teq;
    if (forcing == THOR_FORCING_HELD_SUAREZ) {
      const R day = R(86400.0);
      const R kf = R(1) / day, ka = R(1) / (R(40) * day), ks = R(1) / (R(4) * day);
      const R sb = R(0.7);
      R ramp = div_by(sigma - sb, R(1) - sb, R(1) / (R(1) - sb));
      ramp = ramp > R(0) ? ramp : R(0);
      Kv = kf * ramp;
      R c2 = cl * cl;
      KT = ka + (ks - ka) * ramp * c2 * c2;
      Teq = (R(315) - R(60) * sl * sl - R(10) * lpr * c2) * prk;
      Teq = Teq > R(200) ? Teq : R(200);
    } else {
      const R ss = R(0.12), zs = R(2.0e6);
      const R bt = ld(U.zc + (k)) <= zs ? rsinpi<R>(div_by(sigma - ss, R(2) * (R(1) - ss), R(0.5) / (R(1) - ss))) : R(0);
      Kv = 0;
      KT = R(1) / R(1.5e5);
      Teq = ld(U.hjT + (k)) + bt * (R)hj_dT * clcl;
    }
    // no friction (K_v = 0: above sigma_b, and everywhere on the hot Jupiter)
    // leaves the momentum as it is, so it is neither read nor written there
    if (cmp) {
      if (Kv != R(0)) {
        const R dfr = -Kv * rdt / (R(1) + Kv * rdt);      // 1 / (1 + K_v dt) - 1
        comp_add<R>(X.mx, XL.mx, X.mx, XL.mx, i, (ld(X.mx + i) + ld(XL.mx + i)) * dfr);
        comp_add<R>(X.my, XL.my, X.my, XL.my, i, (ld(X.my + i) + ld(XL.my + i)) * dfr);
        comp_add<R>(X.mz, XL.mz, X.mz, XL.mz, i, (ld(X.mz + i) + ld(XL.mz + i)) * dfr);
      }
      const R dT = KT * rdt * (Teq - Temp) / (R(1) + KT * rdt);
      const R th = ld(U.thb + (k)) + thp;
      comp_add<R>(X.th, XL.th, X.th, XL.th, i, th * rexpm1<R>(rlog1p<R>(dT / Temp) * inv_gamma));
      continue;
    }
    if (Kv != R(0)) {
      R fr = R(1) / (R(1) + Kv * rdt);
      X.mx[i] *= fr;
      X.my[i] *= fr;
      X.mz[i] *= fr;
    }
    if constexpr (sizeof(R) == sizeof(double)) {
      // rho theta at fixed rho scales with T^(1 / gamma); T_new / T - 1 is
      // small (dt over the relaxation time)
      const double y = KT * rdt * (Teq - Temp) / ((1.0 + KT * rdt) * Temp), th = ld(U.thb + (k)) + thp;
      double e;
      if (U.pw && fabs(y) <= 1.0 / 128)
        e = inv_gamma * y * fma(y, fma(y, fma(y, fma(y, fma(y, fma(y, ph.qg[5], ph.qg[4]), ph.qg[3]), ph.qg[2]), ph.qg[1]), ph.qg[0]), 1.0);
      else
        e = pow1p_general(y, inv_gamma).x;
      X.th[i] = fma(th, e, thp);
      continue;
    }
    R Tn = (Temp + KT * rdt * Teq) / (R(1) + KT * rdt);
    // rho theta at fixed rho: Th/Th_bar = ((rho/rho_bar)(T/T_bar))^(1/gamma)
    R lr = rlog1p<R>(rhop / ld(U.rhob + (k))) + rlog<R>(Tn / ld(U.Tb + (k)));
    X.th[i] = ld(U.thb + (k)) * rexpm1<R>(lr * inv_gamma);
  }
}

// ---------------------------------------------------------------- energy budget and fixer
//
// Sec. 3 (after Eq. pressure): an energy fixer after Williamson (2009) that
// adjusts the internal energy by the same amount at every grid point. Once per
// large step (reading F-1) the global diagnostics are reduced at the start of
// the step (fin0) and after the three RK3 stages (fin1); the fixer raises the
// temperature of every cell by dT = (E_start - E_dyn) / (c_v sum V rho) at
// fixed rho and momentum, before the physics. The budget records, per large
// step, mass, energy and axial angular momentum at both points and dT.

// one thread: dT (0 without the fixer) into fix[0] (float64) and fixf[0]
// (storage type), and the step's budget row if recording
template <typename R>
__global__ void k_energy_prepare(const double* fin0, const double* fin1, double cv, int do_fix, double* fix,
                                 R* fixf, double* budget, int* count, int cap) {
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  const double dT = do_fix ? (fin0[1] - fin1[1]) / (cv * fin1[0]) : 0.0;
  fix[0] = dT;
  fixf[0] = (R)dT;
  if (budget) {
    const int n = *count;
    if (n < cap) {
      double* row = budget + (size_t)n * 8;
      row[0] = fin0[0];
      row[1] = fin0[1];
      row[2] = fin0[2];
      row[3] = fin1[0];
      row[4] = fin1[1];
      row[5] = fin1[2];
      row[6] = dT;
      row[7] = 0.0;
      *count = n + 1;
    }
  }
}

// every cell: T -> T + dT at fixed rho, i.e. rho theta (Eq. pressure, in
// deviation form) scaled by (1 + dT / T)^(1 / gamma)
template <typename R>
__global__ void k_energy_fix(Geo<R> G, VR<R> U, Phys ph, Xf<R> X, Xf<R> XL, const R* fixf, int kchunk) {
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= G.ncol) return;
  const int S = G.colp;
  const R dT = ld(fixf);
  const R gamma = pc<R>(ph.gamma, ph.gamma_f), inv_gamma = pc<R>(ph.inv_gamma, ph.inv_gamma_f),
          inv_Rd = pc<R>(ph.inv_Rd, ph.inv_Rd_f);
  const int k0 = blockIdx.y * kchunk, k1 = min(G.nv, k0 + kchunk);
  for (int k = k0; k < k1; ++k) {
    const int i = k * S + c;
    const bool cmp = XL.rho != nullptr;
    const R thp = cmp ? ld(X.th + i) + ld(XL.th + i) : ld(X.th + i);
    const R rho = ld(U.rhob + k) + (cmp ? ld(X.rho + i) + ld(XL.rho + i) : ld(X.rho + i));
    const R p = ld(U.pb + k) + eos_dev<R>(ld(U.pb + k), ld(U.thb + k), thp, gamma);
    const R Temp = p / rho * inv_Rd;
    const R th = ld(U.thb + k) + thp;
    const R d = th * rexpm1<R>(rlog1p<R>(dT / Temp) * inv_gamma);
    if (cmp)
      comp_add<R>(X.th, XL.th, X.th, XL.th, i, d);
    else
      X.th[i] = thp + d;
  }
}

// ---------------------------------------------------------------- kernels: one state

template <typename R, bool HO>
__global__ void k_derived(Geo<R> G, VR<R> U, Phys ph, Xf<R> X, Work<R> T, R* pi, int shallow, int kchunk) {
  d_derived<R, HO>(G, U, ph, X, T, pi, shallow, kchunk, blockIdx.x, blockIdx.y);
}
template <typename R, bool HO>
__global__ void k_lap1(Geo<R> G, VR<R> U, Xf<R> X, Work<R> T, R Kd, int kchunk, int klo, int kend) {
  d_lap1<R, HO>(G, U, X, T, Kd, kchunk, blockIdx.x, blockIdx.y + klo, kend);
}
// DENSE (float): 64 registers and four blocks of 256 threads an SM, one level
// at a time, against 80 and three, two levels at a time. Many cells have threads
// to fill the SMs with (g6 x 32: 64.4 -> 59.3 us, large step 1.202 -> 1.185 ms);
// with fewer the longer threads cost (g5 x 37 22.7 -> 24.6 us, 406 -> 415 us).
template <typename R, bool SH, bool HO, bool DENSE>
__global__ void __launch_bounds__(kMaxBlock, sizeof(R) == sizeof(float) ? (DENSE ? 4 : 3) : 2)
    k_slow(Geo<R> G, VR<R> U, Phys ph, Xf<R> X, Work<R> T, Slow<R> SL, int hyper, R* d0, int kchunk, int klo,
           int kend) {
  d_slow<R, SH, HO, DENSE>(G, U, ph, X, T, SL, hyper, d0, kchunk, blockIdx.x, blockIdx.y + klo, kend);
}
template <typename R, bool HO>
__global__ void k_slow_w(Geo<R> G, VR<R> U, Phys ph, Xf<R> Xt, Xf<R> X, Work<R> T, Slow<R> SL, Pert<R> P, int hyper,
                         int init, int kchunk) {
  d_slow_w<R, HO>(G, U, ph, Xt, X, T, SL, P, hyper, init, kchunk, blockIdx.x, blockIdx.y);
}
template <typename R>
__global__ void k_stage_init(Geo<R> G, VR<R> U, Phys ph, Xf<R> Xt, Xf<R> X, const R* pi, Pert<R> P, Xf<R> XtL,
                             Xf<R> XL, int zero, int kchunk) {
  d_stage_init<R>(G, U, ph, Xt, X, pi, P, XtL, XL, zero, kchunk, blockIdx.x, blockIdx.y);
}
// the small-step stencils take a level range [kchunk * klo, khi) (klo in
// chunks), so that the lower and upper levels can run as separate launches
template <typename R>
__global__ void k_ss_lapd(Geo<R> G, VR<R> U, Work<R> T, const R* dsrc, const R* pstar, R Kd, int kchunk, int klo,
                          int khi) {
  G.nv = khi;
  d_ss_lapd<R>(G, U, T, dsrc, pstar, Kd, kchunk, blockIdx.x, blockIdx.y + klo);
}
// LAST: the last small step of a stage (a separate instantiation, so the
// other small steps carry no registers for the stage end)
template <typename R, bool LAST>
__global__ void k_ss_mom(Geo<R> G, VR<R> U, Slow<R> SL, Pert<R> P, Work<R> T, R dtau, int divdamp,
                         Xf<R> Xs, Xf<R> Xo, Xf<R> XsL, Xf<R> XoL, int kchunk, int klo, int khi) {
  G.nv = khi;
  d_ss_mom<R>(G, U, SL, P, T, dtau, divdamp, Xs, Xo, XsL, XoL, LAST ? 1 : 0, kchunk, blockIdx.x,
              blockIdx.y + klo);
}
template <typename R>
__global__ void k_ss_flux(Geo<R> G, VR<R> U, Slow<R> SL, Pert<R> P, Work<R> T, R dtau, int kchunk, int klo,
                          int khi) {
  G.nv = khi;
  d_ss_flux<R>(G, U, SL, P, T, dtau, kchunk, blockIdx.x, blockIdx.y + klo);
}
// columns and threads of a column kernel's block
template <typename R>
constexpr int col_width() { return sizeof(R) == sizeof(double) ? kCols64 : 32; }
template <typename R>
constexpr int factor_threads() { return sizeof(R) == sizeof(double) ? kThreads64 : 64; }
constexpr int solve_threads() { return 32 * kSolveWarps; }
static_assert(solve_threads() == kThreads64, "one block size for both solves");
template <typename R>
__global__ void __launch_bounds__(factor_threads<R>()) k_ss_factor(Geo<R> G, VR<R> U, Phys ph, Slow<R> SL, Fac<R> F, double dtau) {
  d_ss_factor(G, U, ph, SL, F, dtau, blockIdx.x);
}
template <typename R>
__global__ void __launch_bounds__(32 * kSolveWarps) k_ss_solve(Geo<R> G, VR<R> U, Phys ph, Xf<R> Xs, Slow<R> SL, Pert<R> P,
                                                 Work<R> T, Fac<R> F, double dtau, int want_div, Xf<R> Xo,
                                                 Xf<R> XsL, Xf<R> XoL, int last) {
  d_ss_solve(G, U, ph, Xs, SL, P, T, F, dtau, want_div, Xo, XsL, XoL, last, blockIdx.x);
}
template <typename R>
__global__ void k_surface_p(Geo<R> G, VR<R> U, Phys ph, Xf<R> X, Work<R> T) {
  d_surface_p<R>(G, U, ph, X, T, blockIdx.x);
}
template <typename R>
__global__ void k_physics(Geo<R> G, VR<R> U, Phys ph, Xf<R> X, Xf<R> XL, Work<R> T, int forcing, double dt,
                          double hj_dT, int kchunk) {
  d_physics<R>(G, U, ph, X, XL, T, forcing, dt, hj_dT, kchunk, blockIdx.x, blockIdx.y);
}

// ---------------------------------------------------------------- staged column solve (float storage)
//
// The column step of d_ss_solve for 32 columns with eight warps. Thread 0
// stages the planes of the elimination (W*, S_W, c, a, the matrix's
// off-diagonals, pivot reciprocals, junction factors) into shared memory with
// one cp.async.bulk.tensor per array, and asks the copy engine to prefetch the
// planes of the final updates into L2. All warps then prepare the rows, each
// in its own place: rh_m / piv_m as a double-float product over the pivot
// reciprocal, q over the two off-diagonals, c'/e' over W* and S_W. Warps 0 and
// 1 run the two sweeps and the back substitution, one dependent double-float
// multiply-subtract per row; afterwards all eight warps share the levels of
// Eqs. dens2, pt2 and theta_to_p, whose loads now hit L2. Same operations in
// the same order as d_ss_solve.
// Bound by the memory phases of the blocks resident together (DRAM 39% busy):
// off-diagonals instead of q and c'/e' pairs are 19 words a cell instead of 21
// and 34 KB a block instead of 43, six blocks an SM instead of five (40
// registers, the ensemble's kernel too, which took 64). At g6 x 32 30.8 -> 28.9
// us; 64-member ensemble's large step 11.2 -> 10.6 ms.

// one column group's planes in shared memory (32 columns)
struct SolveSm {
  float *w, *sw, *cc, *ca;        // w: W*, then the solved W*
  float *lo, *up;                 // then q, split into its two words
  float2 *inv;                    // then rh / piv, then d' and f'
  float2 *junc;
  // q and c'/e' of element o (row * 32 + column) after solve_rows
  __device__ float2 q(int o) const { return make_float2(lo[o], up[o]); }
  __device__ float2 cf(int o) const { return make_float2(w[o], sw[o]); }
};
__device__ __forceinline__ SolveSm solve_sm(unsigned char* base, int nv) {
  SolveSm s;
  s.w = reinterpret_cast<float*>(base);             // [nv + 1][32]
  s.sw = s.w + (nv + 1) * 32;                       // [nv + 1][32]
  s.lo = s.sw + (nv + 1) * 32;                      // [nv + 1][32]
  s.up = s.lo + (nv + 1) * 32;                      // [nv + 1][32]
  s.cc = s.up + (nv + 1) * 32;                      // [nv][32]
  s.ca = s.cc + nv * 32;                            // [nv][32]
  s.inv = reinterpret_cast<float2*>(s.ca + nv * 32);  // [nv + 1][32]
  s.junc = s.inv + (nv + 1) * 32;                   // [32]
  return s;
}
// bytes of one group's planes (a multiple of 128, so every plane and what
// follows them starts 128-byte aligned)
__host__ __device__ __forceinline__ size_t solve_stage_bytes(int nv) {
  return (size_t)(4 * (nv + 1) + 2 * nv) * 128 + (size_t)(nv + 2) * 256;
}
size_t solve_tma_smem_bytes(int nv) { return 128 + solve_stage_bytes(nv) + 2 * 256 + sizeof(uint64_t); }

// thread 0 of the copies: the group's elimination planes into s (completing
// on bar) and the planes of its final updates into L2
__device__ __forceinline__ void solve_issue(const SolveSm& s, const SolveMaps& M, int c0, uint64_t* bar, int nv,
                                            int stage0, int want_div) {
  const uint32_t fi = (nv + 1) * 128, fc = nv * 128, di = (nv + 1) * 256;
  const uint64_t ps = pol_stream(), pk = pol_keep();
  mbar_arrive_expect_tx(bar, 4 * fi + 2 * fc + di + 256);
  tma_load_2d(s.w, &M.w, c0, 0, bar, pk);
  tma_load_2d(s.sw, &M.sw, c0, 0, bar, ps);
  tma_load_2d(s.cc, &M.cc, c0, 0, bar, pk);
  tma_load_2d(s.ca, &M.ca, c0, 0, bar, pk);
  tma_load_2d(s.lo, &M.lo, c0, 0, bar, ps);
  tma_load_2d(s.up, &M.up, c0, 0, bar, ps);
  tma_load_2d(s.inv, &M.inv, c0, 0, bar, ps);
  tma_load_2d(s.junc, &M.junction, c0, 0, bar, ps);
  tma_prefetch_2d(&M.thi, c0, 0, ps);
  tma_prefetch_2d(&M.cb, c0, 0, pk);
  tma_prefetch_2d(&M.pi, c0, 0, ps);
  tma_prefetch_2d(stage0 ? &M.th_t : &M.th_s, c0, 0, ps);
  if (want_div) {
    tma_prefetch_2d(&M.dsc, c0, 0, ps);
    tma_prefetch_2d(&M.dhm, c0, 0, pk);
  }
}

// rows m = 1 + warp, + kSolveWarps, ... of one group prepared for the sweeps,
// each row's results over its own inputs (the rows above read only cc and ca)
__device__ __forceinline__ void solve_rows(const SolveSm& s, const VR<float>& U, float rdt, float g, float delta,
                                           int nv, int tx, int warp) {
  const int N = nv - 1, p = N / 2 > 0 ? N / 2 : 1;
  for (int m = 1 + warp; m <= N; m += kSolveWarps) {
    const int o = m * 32 + tx;
    const float wlo = ld(U.wlo + m), whi = ld(U.whi + m);
    const float r = delta * s.w[o] + rdt * s.sw[o] - rdt * ld(U.inv_dzc + m) * (s.cc[o] - s.cc[o - 32])
                    - rdt * g * (wlo * s.ca[o - 32] + whi * s.ca[o]);
    const float2 inv = s.inv[o];
    const float lo = s.lo[o], up = s.up[o];
    const float2 q = df_mul_f(m <= p ? lo : up, inv), cf = df_mul_f(m <= p ? up : lo, inv);
    s.inv[o] = df_product(r, inv);
    s.lo[o] = q.x;
    s.up[o] = q.y;
    s.w[o] = cf.x;
    s.sw[o] = cf.y;
  }
}

// the two sweeps of one group, sweep 0 (rows 1..p, downwards) or 1 (rows
// nv-1..p+1, upwards) by one warp each, then the junction rows and the back
// substitution; the solved W* over s.w. The elimination runs in
// double-float on the float32 pipes. The two warps meet at named barrier 1.
__device__ __forceinline__ void solve_sweeps(const SolveSm& s, float2* sx, int nv, int tx, int sweep) {
  const int N = nv - 1, p = N / 2 > 0 ? N / 2 : 1;
  float2* sdp = s.inv;                                 // rh / piv, then d' / f'
  float* s_wf = s.w;
  if (sweep == 0) {
    float2 d1 = make_float2(0.f, 0.f);
#pragma unroll 4
    for (int m = 1; m <= p; ++m) {
      const int o = m * 32 + tx;
      const float2 r = sdp[o];
      d1 = df_fms(r.x, r.y, s.q(o), d1);
      sdp[o] = d1;
    }
  } else {
    float2 f1 = make_float2(0.f, 0.f);
#pragma unroll 4
    for (int m = N; m > p; --m) {
      const int o = m * 32 + tx;
      const float2 r = sdp[o];
      f1 = df_fms(r.x, r.y, s.q(o), f1);
      sdp[o] = f1;
    }
  }
  asm volatile("bar.sync 1, 64;" ::: "memory");        // the two sweeps only
  if (sweep == 0) {
    const int op = p * 32 + tx;
    float2 xp, xq = make_float2(0.f, 0.f);
    if (p < N) {
      const float2 dp_ = sdp[op], fq = sdp[op + 32];
      xp = df_mul(df_fms(dp_.x, dp_.y, s.cf(op), fq), s.junc[tx]);
      xq = df_fms(fq.x, fq.y, s.cf(op + 32), xp);
    } else {
      xp = sdp[op];
    }
    sx[tx] = xp;
    sx[32 + tx] = xq;
  }
  asm volatile("bar.sync 1, 64;" ::: "memory");
  if (sweep == 0) {
    float2 x = sx[tx];
    s_wf[p * 32 + tx] = df_to_float(x);
    for (int m = p - 1; m >= 1; --m) {
      const int o = m * 32 + tx;
      const float2 d = sdp[o];
      x = df_fms(d.x, d.y, s.cf(o), x);
      s_wf[o] = df_to_float(x);
    }
    s_wf[tx] = 0.f;
  } else {
    float2 x = sx[32 + tx];
    if (p < N) s_wf[(p + 1) * 32 + tx] = df_to_float(x);
    for (int m = p + 2; m <= N; ++m) {
      const int o = m * 32 + tx;
      const float2 d = sdp[o];
      x = df_fms(d.x, d.y, s.cf(o), x);
      s_wf[o] = df_to_float(x);
    }
    s_wf[nv * 32 + tx] = 0.f;
  }
}

// Operands of the final updates (Eqs. dens2, pt2, theta_to_p) of one cell
// that do not depend on the solved W*.
struct UpdOps {
  float thl, thh, cb, pi, ths, dsc, dhm;
};
__device__ __forceinline__ UpdOps upd_load(const Geo<float>& G, const VR<float>& U, const Xf<float>& Xs,
                                           const Slow<float>& SL, const Work<float>& T, int want_div, int k,
                                           int c, uint64_t ps, uint64_t pk) {
  const int nv = G.nv, S = G.colp, i = k * S + c;
  UpdOps o;
  o.thl = k > 0 ? ldh(SL.thi + i, ps) : 0.f;
  o.thh = k + 1 < nv ? ldh(SL.thi + (i + S), ps) : 0.f;
  o.cb = ldh(T.cb + i, pk);
  o.pi = ldh(SL.pi + i, ps);
  o.ths = ld(U.thb + k) + ldh(Xs.th + i, ps);
  o.dsc = want_div ? ldh(SL.dsc + i, ps) : 0.f;
  o.dhm = want_div ? ldh(T.dhm + i, pk) : 0.f;
  return o;
}

// Eqs. dens2, pt2, theta_to_p of one cell with the solved W* (the same
// operations in the same order as d_ss_solve)
__device__ __forceinline__ void upd_apply(const SolveSm& s, const UpdOps& o, const Geo<float>& G,
                                          const VR<float>& U, const Phys& ph, const Xf<float>& Xs,
                                          const Pert<float>& P, const Work<float>& T, float rdt, int want_div,
                                          const Xf<float>& Xo, const Xf<float>& XsL, const Xf<float>& XoL,
                                          int last, int c, int tx, int k, uint64_t pk) {
  const int nv = G.nv, S = G.colp;
  const int q = k * 32 + tx, i = k * S + c;
  const float* s_wf = s.w;
  const float wl = s_wf[q], wh = s_wf[q + 32];
  const float el = ld(U.sq_lo + k), eh = ld(U.sq_hi + k);
  float th_new = o.cb - rdt * (eh * o.thh * wh - el * o.thl * wl);
  const float rho_new = s.ca[q] - rdt * (eh * wh - el * wl);
  sth(P.rho + i, rho_new, pk);
  sth(P.th + i, th_new, pk);
  sth(P.p + i, p_pert(ph, o.pi, o.ths, th_new), pk);
  if (k >= 1) sth(P.w + i, wl, pk);
  if (want_div) sth(T.dd + i, o.dsc + o.dhm + (eh * wh - el * wl), pk);
  if (last) stage_end_cell(Xs, Xo, XsL, XoL, P, rho_new, th_new, wl, k, i, S, nv);
}

// M: the state's descriptors, in kernel-parameter or global memory
__device__ __forceinline__ void d_ss_solve_tma(const Geo<float>& G, const VR<float>& U, const Phys& ph,
                                               const SolveMaps& M, int stage0, const Xf<float>& Xs,
                                               const Slow<float>& SL, const Pert<float>& P, const Work<float>& T,
                                               double dtau, int want_div, const Xf<float>& Xo, const Xf<float>& XsL,
                                               const Xf<float>& XoL, int last, int* err, int bx) {
  extern __shared__ unsigned char smraw[];
  const int nv = G.nv;
  const int tid = threadIdx.x, tx = tid & 31, warp = tid >> 5;
  unsigned char* base = smraw + ((128u - (smem_u32(smraw) & 127u)) & 127u);
  const SolveSm s = solve_sm(base, nv);
  float2* sx = reinterpret_cast<float2*>(base + solve_stage_bytes(nv));   // [2][32]
  uint64_t* bar = reinterpret_cast<uint64_t*>(sx + 64);

  if (tid == 0) {
    mbar_init(bar, 1);
    mbar_init_fence();
  }
  pdl_next();
  const int c0 = pdl_wait(bx * 32), c = c0 + tx;
  __syncthreads();
  if (tid == 0) solve_issue(s, M, c0, bar, nv, stage0, want_div);
  if (!__syncthreads_and(mbar_wait(bar, 0))) {
    if (tid == 0) {                      // flag, give the copies a bounded time to land, leave
      atomicExch(err, 1);
      mbar_wait(bar, 0);
    }
    return;
  }
  const float rdt = (float)dtau, g = ph.g_f;
  solve_rows(s, U, rdt, g, ph.delta_f, nv, tx, warp);
  __syncthreads();
  if (warp < 2) solve_sweeps(s, sx, nv, tx, warp);
  __syncthreads();
  if (c >= G.ncol) return;
  // the eight warps share the levels of the final updates
  const uint64_t ps = pol_stream(), pk = pol_keep();
#pragma unroll 4
  for (int k = warp; k < nv; k += kSolveWarps)
    upd_apply(s, upd_load(G, U, Xs, SL, T, want_div, k, c, ps, pk), G, U, ph, Xs, P, T, rdt, want_div, Xo, XsL,
              XoL, last, c, tx, k, pk);
}

__global__ void __launch_bounds__(32 * kSolveWarps, 6)
    k_ss_solve_tma(Geo<float> G, VR<float> U, Phys ph, const __grid_constant__ SolveMaps M, int stage0,
                   Xf<float> Xs, Slow<float> SL, Pert<float> P, Work<float> T, double dtau, int want_div,
                   Xf<float> Xo, Xf<float> XsL, Xf<float> XoL, int last, int* err) {
  d_ss_solve_tma(G, U, ph, M, stage0, Xs, SL, P, T, dtau, want_div, Xo, XsL, XoL, last, err, blockIdx.x);
}

// ---------------------------------------------------------------- kernels: ensemble
//
// One launch covers every member: block b of the launch works on local block
// map[b].y of member map[b].x, whose arrays and constants come from the
// member table. Per-member switches (hyperdiffusion, divergence damping,
// forcing) are uniform over a block. s is the RK stage, j the small step.

// The block's member record is copied to shared memory once, and the device
// functions read its fields from there as they need them (by reference), so
// that the record's pointers do not all occupy registers. The copy (1.3 KB and
// a barrier) costs a block as much as a level of its stencils, so the stencil
// blocks hold 256 threads: 256 columns by default, or, where the block is tuned to
// fewer columns, several level chunks of them (threadIdx.y; 64
// members at 8 levels a thread, 256 / 128 / 64 columns: 11.17 / 11.15 / 12.11 ms a step).
template <typename T>
__device__ __forceinline__ const T& stage_record(const T* src, T* dst) {
  static_assert(sizeof(T) % 4 == 0, "record of whole words");
  const uint32_t* a = reinterpret_cast<const uint32_t*>(src);
  uint32_t* b = reinterpret_cast<uint32_t*>(dst);
  for (int w = threadIdx.y * blockDim.x + threadIdx.x; w < (int)(sizeof(T) / 4); w += blockDim.x * blockDim.y) b[w] = a[w];
  __syncthreads();
  return *dst;
}

// the level chunk of a thread of the stencil kernels
__device__ __forceinline__ int member_chunk() { return blockIdx.y * blockDim.y + threadIdx.y; }

#define THOR_MEMBER()                                   \
  __shared__ Member<R> a_sm;                            \
  const int2 e = map[blockIdx.x];                       \
  const Member<R>& a = stage_record(M + e.x, &a_sm);    \
  const Xf<R>& Xs = s == 0 ? a.Xt : a.Xst

template <typename R>
__global__ void ke_derived(const Member<R>* __restrict__ M, const int2* __restrict__ map, int s, int kchunk) {
  THOR_MEMBER();
  if (a.ph.vorder > 1)
    d_derived<R, true>(a.G, a.U, a.ph, Xs, a.T, a.SL.pi, a.shallow, kchunk, e.y, member_chunk());
  else
    d_derived<R>(a.G, a.U, a.ph, Xs, a.T, a.SL.pi, a.shallow, kchunk, e.y, member_chunk());
}
template <typename R>
__global__ void ke_lap1(const Member<R>* __restrict__ M, const int2* __restrict__ map, int s, int kchunk) {
  THOR_MEMBER();
  if (a.hyper && a.ph.vorder > 1)
    d_lap1<R, true>(a.G, a.U, Xs, a.T, a.Kd, kchunk, e.y, member_chunk(), a.G.nv + 1);
  else if (a.hyper)
    d_lap1<R>(a.G, a.U, Xs, a.T, a.Kd, kchunk, e.y, member_chunk(), a.G.nv + 1);
}
template <typename R>
__global__ void __launch_bounds__(kMaxBlock, 2)
    ke_slow(const Member<R>* __restrict__ M, const int2* __restrict__ map, int s, int kchunk) {
  THOR_MEMBER();
  R* d0 = s == 0 && a.divdamp ? a.T.dd0 : nullptr;
  const bool ho = a.ph.vorder > 1;
  if (a.shallow && ho)
    d_slow<R, true, true>(a.G, a.U, a.ph, Xs, a.T, a.SL, a.hyper, d0, kchunk, e.y, member_chunk(), a.G.nv);
  else if (a.shallow)
    d_slow<R, true>(a.G, a.U, a.ph, Xs, a.T, a.SL, a.hyper, d0, kchunk, e.y, member_chunk(), a.G.nv);
  else if (ho)
    d_slow<R, false, true>(a.G, a.U, a.ph, Xs, a.T, a.SL, a.hyper, d0, kchunk, e.y, member_chunk(), a.G.nv);
  else
    d_slow<R, false>(a.G, a.U, a.ph, Xs, a.T, a.SL, a.hyper, d0, kchunk, e.y, member_chunk(), a.G.nv);
}
template <typename R>
__global__ void ke_slow_w(const Member<R>* __restrict__ M, const int2* __restrict__ map, int s, int kchunk) {
  THOR_MEMBER();
  const Xf<R> XtL = s == 0 ? Xf<R>{} : a.XtL;      // stage 0: X^(s) is X^t, pair and all
  if (a.ph.vorder > 1)
    d_slow_w<R, true>(a.G, a.U, a.ph, a.Xt, Xs, a.T, a.SL, a.P, a.hyper, 1, kchunk, e.y, member_chunk(), XtL);
  else
    d_slow_w<R>(a.G, a.U, a.ph, a.Xt, Xs, a.T, a.SL, a.P, a.hyper, 1, kchunk, e.y, member_chunk(), XtL);
}
template <typename R>
__global__ void __launch_bounds__(factor_threads<R>())
    ke_ss_factor(const Member<R>* __restrict__ M, const int2* __restrict__ map, int s) {
  THOR_MEMBER();
  d_ss_factor(a.G, a.U, a.ph, a.SL, a.F, a.dts[s], e.y);
}
template <typename R>
// the small-step stencils over levels [kchunk * klo, khi) (as k_ss_*)
__global__ void ke_ss_lapd(const Member<R>* __restrict__ M, const int2* __restrict__ map, int s, int j,
                           int kchunk, int klo, int khi) {
  THOR_MEMBER();
  Geo<R> G = a.G;
  G.nv = khi;
  if (a.divdamp) d_ss_lapd<R>(G, a.U, a.T, j == 0 ? a.T.dd0 : a.T.dd, a.P.p, a.Kd, kchunk, e.y, member_chunk() + klo);
}
template <typename R>
__global__ void ke_ss_mom(const Member<R>* __restrict__ M, const int2* __restrict__ map, int s, int j,
                          int kchunk, int klo, int khi) {
  THOR_MEMBER();
  Geo<R> G = a.G;
  G.nv = khi;
  d_ss_mom<R>(G, a.U, a.SL, a.P, a.T, (R)a.dts[s], a.divdamp, Xs, s == 2 ? a.Xt : a.Xst,
              s == 0 ? a.XtL : Xf<R>{}, s == 2 ? a.XtL : Xf<R>{}, j + 1 == a.nsub[s], kchunk, e.y,
              member_chunk() + klo);
}
template <typename R>
__global__ void ke_ss_flux(const Member<R>* __restrict__ M, const int2* __restrict__ map, int s, int kchunk,
                           int klo, int khi) {
  THOR_MEMBER();
  Geo<R> G = a.G;
  G.nv = khi;
  d_ss_flux<R>(G, a.U, a.SL, a.P, a.T, (R)a.dts[s], kchunk, e.y, member_chunk() + klo);
}
template <typename R>
__global__ void __launch_bounds__(32 * kSolveWarps)
    ke_ss_solve(const Member<R>* __restrict__ M, const int2* __restrict__ map, int s, int j) {
  THOR_MEMBER();
  const int want_div = a.divdamp && j + 1 < a.nsub[s];
  d_ss_solve(a.G, a.U, a.ph, Xs, a.SL, a.P, a.T, a.F, a.dts[s], want_div, s == 2 ? a.Xt : a.Xst,
             s == 0 ? a.XtL : Xf<R>{}, s == 2 ? a.XtL : Xf<R>{}, j + 1 == a.nsub[s], e.y);
}
__global__ void __launch_bounds__(32 * kSolveWarps, 6)
    ke_ss_solve_tma(const Member<float>* __restrict__ M, const int2* __restrict__ map, int s, int j) {
  const int2 e = map[blockIdx.x];
  const Member<float>& a = M[e.x];
  const Xf<float> Xs = s == 0 ? a.Xt : a.Xst;
  const int want_div = a.divdamp && j + 1 < a.nsub[s];
  d_ss_solve_tma(a.G, a.U, a.ph, *a.smap, s == 0, Xs, a.SL, a.P, a.T, a.dts[s], want_div, s == 2 ? a.Xt : a.Xst,
                 s == 0 ? a.XtL : Xf<float>{}, s == 2 ? a.XtL : Xf<float>{}, j + 1 == a.nsub[s], a.err, e.y);
}
template <typename R>
__global__ void ke_surface_p(const Member<R>* __restrict__ M, const int2* __restrict__ map) {
  const int2 e = map[blockIdx.x];
  const Member<R>& a = M[e.x];
  if (a.forcing) d_surface_p<R>(a.G, a.U, a.ph, a.Xt, a.T, e.y);
}
template <typename R>
__global__ void ke_physics(const Member<R>* __restrict__ M, const int2* __restrict__ map, int kchunk) {
  const int2 e = map[blockIdx.x];
  const Member<R>& a = M[e.x];
  if (a.forcing) d_physics<R>(a.G, a.U, a.ph, a.Xt, a.XtL, a.T, a.forcing, a.dt, a.hj_dT, kchunk, e.y, blockIdx.y);
}
#undef THOR_MEMBER

// ---------------------------------------------------------------- driver

template <typename R>
void Impl<R>::launch_2d(int nplanes, int kchunk, dim3& grid) const {
  grid = dim3((G.ncol + block - 1) / block, (nplanes + kchunk - 1) / kchunk);
}

template <typename R>
size_t solve_smem_bytes(int nv) {
  return (size_t)(2 * (nv + 1) + (sizeof(R) == sizeof(float) ? 2 : 0)) * col_width<R>() * sizeof(double);
}
template <typename R>
size_t factor_smem_bytes(int nv) {
  return sizeof(R) == sizeof(double) ? (size_t)3 * (nv + 1) * kCols64 * sizeof(double) : 0;
}
template <typename R>
int column_width() { return col_width<R>(); }
template int column_width<double>();
template int column_width<float>();

// Raise a kernel's dynamic shared-memory limit to at least bytes, never
// lower it: states with different level counts share the kernels, and a
// later state with fewer levels must not take room from an earlier one.
template <typename K>
static bool raise_smem_limit(K* kernel, int bytes) {
  cudaFuncAttributes a{};
  if (cudaFuncGetAttributes(&a, kernel) != cudaSuccess) return false;
  if (a.maxDynamicSharedSizeBytes >= bytes) return true;
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes) == cudaSuccess;
}

template <typename R>
int col_kernel_setup(int nv) {
  const int bytes = (int)solve_smem_bytes<R>(nv), fbytes = (int)factor_smem_bytes<R>(nv);
  return raise_smem_limit(k_ss_solve<R>, bytes) && raise_smem_limit(ke_ss_solve<R>, bytes) &&
                 raise_smem_limit(k_ss_factor<R>, fbytes) && raise_smem_limit(ke_ss_factor<R>, fbytes)
             ? 0
             : -3;
}
template int col_kernel_setup<double>(int);
template int col_kernel_setup<float>(int);

// the slow-term kernel of a state
template <typename R, bool DENSE>
auto slow_kernel(bool shallow, bool ho) {
  return shallow ? (ho ? k_slow<R, true, true, DENSE> : k_slow<R, true, false, DENSE>)
                 : (ho ? k_slow<R, false, true, DENSE> : k_slow<R, false, false, DENSE>);
}
template <typename R>
auto slow_kernel(bool shallow, bool ho, bool dense) {
  if constexpr (sizeof(R) == sizeof(float))
    if (dense) return slow_kernel<R, true>(shallow, ho);
  return slow_kernel<R, false>(shallow, ho);
}

template <typename R>
int Impl<R>::large_step(double dt, int n_small) {
  const int kc = kchunk, bs = block;
  dim3 g2, g2i;
  launch_2d(G.nv, kc, g2);
  launch_2d(G.nv + 1, kc, g2i);
  dim3 g1((G.ncol + bs - 1) / bs);
  dim3 gsolve((G.ncol + col_width<R>() - 1) / col_width<R>());
  const size_t solve_smem = solve_smem_bytes<R>(G.nv);
  const bool staged = solve_tma && smaps != nullptr;
  // level halves of the small-step stencils (THOR_TUNE_LEVEL_SPLIT): levels
  // [0, kc * hc) on the state's stream, [kc * hc, nv) on side2
  const bool lsplit = level_split && side != nullptr && !prof_on && side2 != nullptr && G.nv >= 2 * kc;
  const bool pdl = overlap && !lsplit && !prof_on && stream != nullptr && (long long)g2.x * g2.y <= sms;
  auto hint = [&](bool after) { return LaunchHint{after, carveout}; };
  const int nch = (G.nv + kc - 1) / kc, hc = lsplit ? nch / 2 : nch;
  dim3 glo(g2.x, hc), ghi(g2.x, nch - hc);
  const R Kd = (R)(diff_D * dbar4 / dt);
  auto lapd = [&](bool after, cudaStream_t st, const R* dsrc, dim3 g, int klo, int khi) -> cudaError_t {
    return launch_hint(hint(after), k_ss_lapd<R>, g, bs, 0, st, G, U, T, dsrc, (const R*)P.p, Kd, kc, klo, khi);
  };
  const double dts[3] = {dt / 3.0, dt / n_small, dt / n_small};
  const int nsub[3] = {1, n_small / 2, n_small};
  cudaError_t e = cudaSuccess;
  auto chk = [&](cudaError_t r) {
    if (e == cudaSuccess) e = r;
  };
  // Kernels of a stage that do not depend on each other run on two streams
  // (graph branches when captured): after k_derived the stage's perturbations
  // (k_stage_init) and, from the second stage on, the first small step's
  // gradient of D (of X^t, kept from the first stage) run on the side stream
  // beside the slow terms; after k_slow_w the factorisation runs there beside
  // the first small step's stencils. With per-kernel profiling everything
  // stays on the state's stream, in the same order.
  const bool fork = side != nullptr && !prof_on;
  const int nstages = rk_stages;      // 3, or fewer when a test stops the step early
  const bool energy = (energy_fix || budget_cap > 0) && fixbuf != nullptr && nstages == 3;
  double* fin0 = fixbuf + kDiagBlocks * 8;                       // reduction at the step start
  double* part1 = fixbuf + (kDiagBlocks + 1) * 8;
  double* fin1 = part1 + kDiagBlocks * 8;                        // after the dynamics
  double* fixv = fin1 + 8;
  R* fixf = reinterpret_cast<R*>(fixv + 1);
  if (energy) {
    chk(launch_k(k_diag_partial<R>, kDiagBlocks, kDiagThreads, 0, stream, G, V, ph, Xt, XtL, fixbuf));
    chk(launch_k(k_diag_final, 1, 256, 0, stream, fixbuf, kDiagBlocks));
    launches += 2;
  }
  for (int s = 0; s < nstages; ++s) {
    // the last stage run writes X^(s+1) into the state
    Xf<R> Xs = s == 0 ? Xt : Xst, Xo = s == nstages - 1 ? Xt : Xst;
    // low parts of a compensated state: X^t keeps them; a stage state is
    // stored as floats (the next stage's perturbations start from the stored
    // value, so its rounding cancels at the last stage end, which writes X^t
    // as a pair)
    Xf<R> XsL = s == 0 ? XtL : Xf<R>{}, XoL = s == nstages - 1 ? XtL : Xf<R>{};
    cudaStream_t aux = fork ? side : stream;
    mark(THOR_K_DERIVED, true);
    const bool ho = ph.vorder > 1;
    chk(launch_hint(hint(pdl && s > 0), ho ? k_derived<R, true> : k_derived<R, false>, g2i, bs, 0, stream, G, U, ph, Xs, T, SL.pi, shallow, kc));
    mark(THOR_K_DERIVED, false);
    ++launches;
    if (fork) {
      chk(cudaEventRecord(ev_fork, stream));
      chk(cudaStreamWaitEvent(side, ev_fork, 0));
    }
    mark(THOR_K_STAGE_INIT, true);
    chk(launch_hint(hint(false), k_stage_init<R>, g2i, bs, 0, aux, G, U, ph, Xt, Xs, (const R*)SL.pi, P, XtL, XsL, (int)(s == 0), kc));
    mark(THOR_K_STAGE_INIT, false);
    ++launches;
    const bool early_grad = divdamp && s > 0;    // D of X^t is ready before the slow terms
    if (early_grad) {
      mark(THOR_K_SS_LAPD, true);
      chk(lapd(pdl, aux, (const R*)T.dd0, g2, 0, G.nv));
      mark(THOR_K_SS_LAPD, false);
      ++launches;
    }
    if (fork) chk(cudaEventRecord(ev_join0, side));
    if (hyper) {
      mark(THOR_K_LAP1, true);
      chk(launch_hint(hint(pdl), ho ? k_lap1<R, true> : k_lap1<R, false>, g2i, bs, 0, stream, G, U, Xs, T, Kd, kc, 0, G.nv + 1));
      mark(THOR_K_LAP1, false);
      ++launches;
    }
    mark(THOR_K_SLOW, true);
    auto slow = slow_kernel<R>(shallow, ho, dense);
    chk(launch_hint(hint(pdl), slow, g2, bs, 0, stream, G, U, ph, Xs, T, SL, hyper,
                 s == 0 && divdamp ? T.dd0 : (R*)nullptr, kc, 0, G.nv));
    mark(THOR_K_SLOW, false);
    ++launches;
    // the vertical momentum's slow term and the factorisation only gate the
    // first column solve: they run on the side stream beside the first
    // small step's stencils
    if (fork) {
      chk(cudaEventRecord(ev_fork, stream));
      chk(cudaStreamWaitEvent(side, ev_fork, 0));
    }
    mark(THOR_K_SLOW_W, true);
    chk(launch_hint(hint(false), ho ? k_slow_w<R, true> : k_slow_w<R, false>, g2i, bs, 0, aux, G, U, ph, Xt, Xs, T, SL, P, hyper, 0,
                 kc));
    mark(THOR_K_SLOW_W, false);
    mark(THOR_K_SS_FACTOR, true);
    chk(launch_hint(hint(pdl), k_ss_factor<R>, gsolve, factor_threads<R>(), factor_smem_bytes<R>(G.nv), aux, G, U, ph, SL, F, dts[s]));
    mark(THOR_K_SS_FACTOR, false);
    if (fork) {
      chk(cudaEventRecord(ev_join, side));
      chk(cudaStreamWaitEvent(stream, ev_join0, 0));
    }
    launches += 2;
    for (int j = 0; j < nsub[s]; ++j) {
      // the last small step of a stage also ends the stage: X^(s+1) = X^(s) + X*
      const int last = j + 1 == nsub[s];
      // the three horizontal stencils over levels [kc * klo, khi) on st
      auto stencils = [&](cudaStream_t st, dim3 g, int klo, int khi) {
        // D: of X^t in the first small step, then from the previous column step
        if (divdamp && !(j == 0 && early_grad)) {
          mark(THOR_K_SS_LAPD, true);
          chk(lapd(pdl && j > 0, st, (const R*)(j == 0 ? T.dd0 : T.dd), g, klo, khi));
          mark(THOR_K_SS_LAPD, false);
          ++launches;
        }
        mark(THOR_K_SS_MOM, true);
        chk(launch_hint(hint(pdl && (j > 0 || (divdamp && !early_grad))), last ? k_ss_mom<R, true> : k_ss_mom<R, false>, g, bs, 0, st, G, U, SL, P, T, (R)dts[s],
                     divdamp, Xs, Xo, XsL, XoL, kc, klo, khi));
        mark(THOR_K_SS_MOM, false);
        mark(THOR_K_SS_FLUX, true);
        chk(launch_hint(hint(pdl), k_ss_flux<R>, g, bs, 0, st, G, U, SL, P, T, (R)dts[s], kc, klo, khi));
        mark(THOR_K_SS_FLUX, false);
        launches += 2;
      };
      if (lsplit) {
        chk(cudaEventRecord(ev_s1, stream));
        chk(cudaStreamWaitEvent(side2, ev_s1, 0));
        stencils(stream, glo, 0, kc * hc);
        stencils(side2, ghi, hc, G.nv);
        chk(cudaEventRecord(ev_s2, side2));
        chk(cudaStreamWaitEvent(stream, ev_s2, 0));
      } else {
        stencils(stream, g2, 0, G.nv);
      }
      const int want_div = divdamp && !last;
      if (fork && j == 0) chk(cudaStreamWaitEvent(stream, ev_join, 0));
      mark(THOR_K_SS_SOLVE, true);
      if (staged)
        chk(launch_solve_tma(hint(pdl && j > 0), gsolve, s, Xo, XsL, XoL, dts[s], want_div, last));
      else
        chk(launch_hint(hint(pdl && j > 0), k_ss_solve<R>, gsolve, solve_threads(), solve_smem, stream, G, U, ph, Xs, SL, P, T, F, dts[s],
                     want_div, Xo, XsL, XoL, last));
      mark(THOR_K_SS_SOLVE, false);
      ++launches;
    }
  }
  if (energy) {
    chk(launch_k(k_diag_partial<R>, kDiagBlocks, kDiagThreads, 0, stream, G, V, ph, Xt, XtL, part1));
    chk(launch_k(k_diag_final, 1, 256, 0, stream, part1, kDiagBlocks));
    chk(launch_k(k_energy_prepare<R>, 1, 32, 0, stream, (const double*)fin0, (const double*)fin1, ph.cv,
                 energy_fix, fixv, fixf, budget_cap > 0 ? budget : (double*)nullptr, budget_count, budget_cap));
    launches += 3;
    if (energy_fix) {
      chk(launch_k(k_energy_fix<R>, g2, bs, 0, stream, G, U, ph, Xt, XtL, (const R*)fixf, kc));
      ++launches;
    }
  }
  if (forcing != 0 && nstages == 3) {
    mark(THOR_K_PHYSICS, true);
    chk(launch_hint(hint(pdl && !energy), k_surface_p<R>, g1, bs, 0, stream, G, U, ph, Xt, T));
    chk(launch_hint(hint(pdl), k_physics<R>, g2, bs, 0, stream, G, U, ph, Xt, XtL, T, forcing, dt, hj_dT, kc));
    mark(THOR_K_PHYSICS, false);
    launches += 2;
  }
  return e == cudaSuccess && cudaGetLastError() == cudaSuccess ? 0 : -3;
}

template <typename R>
int anelastic_project(Impl<R>& I, double dts, const Xf<R>& Xo, int* iters);   // thor_anelastic.cu

// One large step under the anelastic switch (Sec. 3): the three RK3 stages
// of lengths dt/3, dt/2, dt, each the slow terms at the stage state
// (pressure gradient and gravity replaced by the buoyancy) and one
// projection from X^t (thor_anelastic.cu), then the physics.
template <typename R>
int Impl<R>::anelastic_step(double dt) {
  const int kc = kchunk, bs = block;
  dim3 g2, g2i;
  launch_2d(G.nv, kc, g2);
  launch_2d(G.nv + 1, kc, g2i);
  dim3 g1((G.ncol + bs - 1) / bs);
  const R Kd = (R)(diff_D * dbar4 / dt);
  const double dts[3] = {dt / 3.0, dt / 2.0, dt};
  const bool ho = ph.vorder > 1;
  for (int s = 0; s < 3; ++s) {
    Xf<R> Xs = s == 0 ? Xt : Xst, Xo = s == 2 ? Xt : Xst;
    if (launch_k(ho ? k_derived<R, true> : k_derived<R, false>, g2i, bs, 0, stream, G, U, ph, Xs, T, SL.pi, shallow, kc))
      return -3;
    if (hyper && launch_k(ho ? k_lap1<R, true> : k_lap1<R, false>, g2i, bs, 0, stream, G, U, Xs, T, Kd, kc, 0,
                          G.nv + 1))
      return -3;
    auto slow = slow_kernel<R>(shallow, ho, dense);
    if (launch_k(slow, g2, bs, 0, stream, G, U, ph, Xs, T, SL, hyper, (R*)nullptr, kc, 0, G.nv) ||
        launch_k(ho ? k_slow_w<R, true> : k_slow_w<R, false>, g2i, bs, 0, stream, G, U, ph, Xt, Xs, T, SL, P,
                 hyper, 0, kc))
      return -3;
    launches += 3 + (hyper ? 1 : 0);
    int it = 0;
    const int rc = anelastic_project(*this, dts[s], Xo, &it);
    an_last_iters = it;
    if (rc) return rc;
  }
  if (forcing != 0) {
    if (launch_k(k_surface_p<R>, g1, bs, 0, stream, G, U, ph, Xt, T) ||
        launch_k(k_physics<R>, g2, bs, 0, stream, G, U, ph, Xt, XtL, T, forcing, dt, hj_dT, kc))
      return -3;
    launches += 2;
  }
  return cudaGetLastError() == cudaSuccess ? 0 : -3;
}
template int Impl<double>::anelastic_step(double);
template int Impl<float>::anelastic_step(double);

template <>
cudaError_t Impl<float>::launch_solve_tma(LaunchHint hint, dim3 grid, int stage, const Xf<float>& Xo, const Xf<float>& XsL,
                                          const Xf<float>& XoL, double dtau, int want_div, int last) {
  return launch_hint(hint, k_ss_solve_tma, grid, 32 * kSolveWarps, solve_tma_smem_bytes(G.nv), stream, G, U, ph, *smaps,
                  (int)(stage == 0), stage == 0 ? Xt : Xst, SL, P, T, dtau, want_div, Xo, XsL, XoL, last, dev_err);
}
template <>
cudaError_t Impl<double>::launch_solve_tma(LaunchHint, dim3, int, const Xf<double>&, const Xf<double>&, const Xf<double>&,
                                           double, int, int) {
  return cudaErrorInvalidValue;
}

// TMA descriptors of the staged solve (float storage only; the float64
// planes would not fit the shared memory of a useful number of blocks)
template <>
int Impl<float>::build_solve_maps() {
  static void* encode_fn = nullptr;
  const size_t smem = solve_tma_smem_bytes(G.nv);
  if (smem > 200 * 1024) return 0;                  // stays on the direct solve
  if (!encode_fn) {
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &encode_fn, 12000, cudaEnableDefault, &q) !=
            cudaSuccess ||
        q != cudaDriverEntryPointSuccess || !encode_fn) {
      encode_fn = nullptr;
      return 0;
    }
  }
  using Encode = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                              const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                              CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
  Encode encode = reinterpret_cast<Encode>(encode_fn);
  auto map = std::make_unique<SolveMaps>();
  bool ok = true;
  auto make = [&](CUtensorMap* m, const void* ptr, int planes, bool dbl) {
    const cuuint64_t dims[2] = {(cuuint64_t)G.colp, (cuuint64_t)planes};
    const cuuint64_t strides[1] = {(cuuint64_t)G.colp * (dbl ? 8 : 4)};
    const cuuint32_t box[2] = {32, (cuuint32_t)planes};
    const cuuint32_t es[2] = {1, 1};
    ok = ok && encode(m, dbl ? CU_TENSOR_MAP_DATA_TYPE_FLOAT64 : CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2,
                      const_cast<void*>(ptr), dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
                      CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_NONE,
                      CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
  };
  const int nv = G.nv;
  make(&map->w, P.w, nv + 1, false);
  make(&map->sw, SL.sw, nv + 1, false);
  make(&map->thi, SL.thi, nv + 1, false);
  make(&map->cc, T.cc, nv, false);
  make(&map->ca, T.ca, nv, false);
  make(&map->cb, T.cb, nv, false);
  make(&map->pi, SL.pi, nv, false);
  make(&map->th_t, Xt.th, nv, false);
  make(&map->th_s, Xst.th, nv, false);
  make(&map->dsc, SL.dsc, nv, false);
  make(&map->dhm, T.dhm, nv, false);
  make(&map->lo, F.q, nv + 1, false);
  make(&map->up, F.cf, nv + 1, false);
  make(&map->inv, F.inv, nv + 1, true);
  make(&map->junction, F.junction, 1, true);
  if (!ok) return 0;
  if (!raise_smem_limit(k_ss_solve_tma, (int)smem) || !raise_smem_limit(ke_ss_solve_tma, (int)smem)) return -3;
  smaps = std::move(map);
  return 0;
}
template <>
int Impl<double>::build_solve_maps() {
  return 0;
}

template void Impl<double>::launch_2d(int, int, dim3&) const;
template void Impl<float>::launch_2d(int, int, dim3&) const;
template int Impl<double>::large_step(double, int);
template int Impl<float>::large_step(double, int);

// One large step of every member of an ensemble, one launch per kernel of
// the sequence above. Members are ordered by decreasing n_small, so the
// members still in their small-step loop at step j of a stage are a prefix
// of the block maps.
template <typename R>
int ensemble_large_step(const EnsPlan<R>& E, cudaStream_t stream, long long* launches) {
  const int kc = E.kchunk, bs = E.block;
  const int yc = (E.nv + kc - 1) / kc, yci = (E.nv + 1 + kc - 1) / kc;
  // blocks of bs columns x rows level chunks
  const int rows = max(1, kMaxBlock / bs);
  const dim3 tb(bs, rows);
  auto up = [&](int chunks) { return (chunks + rows - 1) / rows; };
  const size_t solve_smem = solve_smem_bytes<R>(E.nv);
  const Member<R>* M = E.M;
  long long n = 0;
  for (int s = 0; s < 3; ++s) {
    const dim3 g2(E.nblk, up(yc)), g2i(E.nblk, up(yci));
    ke_derived<R><<<g2i, tb, 0, stream>>>(M, E.map, s, kc);
    if (E.any_hyper) {
      ke_lap1<R><<<g2i, tb, 0, stream>>>(M, E.map, s, kc);
      ++n;
    }
    ke_slow<R><<<g2, tb, 0, stream>>>(M, E.map, s, kc);
    ke_slow_w<R><<<g2i, tb, 0, stream>>>(M, E.map, s, kc);
    ke_ss_factor<R><<<E.nblkc, factor_threads<R>(), factor_smem_bytes<R>(E.nv), stream>>>(M, E.mapc, s);
    n += 4;
    for (int j = 0; j < E.maxsub[s]; ++j) {
      const int nb = E.active[s][j], nbc = E.activec[s][j];
      // the stencils over level chunks [c0, c1) on st
      auto stencils = [&](cudaStream_t st, int c0, int c1) {
        const dim3 a2(nb, up(c1 - c0));
        const int khi = min(E.nv, c1 * kc);
        if (E.any_divdamp) {
          ke_ss_lapd<R><<<a2, tb, 0, st>>>(M, E.map, s, j, kc, c0, khi);
          ++n;
        }
        ke_ss_mom<R><<<a2, tb, 0, st>>>(M, E.map, s, j, kc, c0, khi);
        ke_ss_flux<R><<<a2, tb, 0, st>>>(M, E.map, s, kc, c0, khi);
        n += 2;
      };
      if (E.side2 && yc >= 2) {
        cudaEventRecord(E.ev_a, stream);
        cudaStreamWaitEvent(E.side2, E.ev_a, 0);
        stencils(stream, 0, yc / 2);
        stencils(E.side2, yc / 2, yc);
        cudaEventRecord(E.ev_b, E.side2);
        cudaStreamWaitEvent(stream, E.ev_b, 0);
      } else {
        stencils(stream, 0, yc);
      }
      if constexpr (sizeof(R) == sizeof(float)) {
        if (E.staged)
          ke_ss_solve_tma<<<nbc, 32 * kSolveWarps, solve_tma_smem_bytes(E.nv), stream>>>(M, E.mapc, s, j);
        else
          ke_ss_solve<R><<<nbc, 32 * kSolveWarps, solve_smem, stream>>>(M, E.mapc, s, j);
      } else {
        ke_ss_solve<R><<<nbc, 32 * kSolveWarps, solve_smem, stream>>>(M, E.mapc, s, j);
      }
      ++n;
    }
  }
  if (E.any_forcing) {
    ke_surface_p<R><<<E.nblk, bs, 0, stream>>>(M, E.map);
    ke_physics<R><<<dim3(E.nblk, yc), bs, 0, stream>>>(M, E.map, kc);
    n += 2;
  }
  *launches += n;
  return cudaGetLastError() == cudaSuccess ? 0 : -3;
}

template int ensemble_large_step<double>(const EnsPlan<double>&, cudaStream_t, long long*);
template int ensemble_large_step<float>(const EnsPlan<float>&, cudaStream_t, long long*);

}  // namespace thor
