// Zonal band means of a state on the GPU (Sec. 6.1: the Held-Suarez and
// hot-Jupiter climates are judged by zonal and time averages of the wind and
// temperature, the mass stream function and the eddy fluxes [u'v'], [v'T']).
//
// A zonal mean on the icosahedral grid is the volume-weighted mean over the
// cells of one level whose latitude falls in one of nlat equal bands (band
// b = floor((lat + pi/2 + 1e-9) / pi * nlat), the north pole in the last
// band).
// thor_zonal_accumulate reduces the current state to per-(level, band) sums
// of V, V u, V v, V T, V p, V uv, V vT, V uu, V vv (float64), turns them into the
// band means and covariances of that state and adds them to the state's
// time accumulator; thor_zonal_read returns the accumulated sums. At the two
// polar cells east and north are undefined and u = v = 0. The same pass adds
// every cell's vertical velocity at its centre, w = (W interpolated to the
// centre) / rho, to a per-cell time sum: the time mean [w] behind the
// grid-imprinting map [w*] of Sec. 6.1 (thor_zonal_read_w).
#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "../../include/thor.h"
#include "thor_state.h"

namespace thor {
namespace {

// One block sums one chunk of a band's columns (ZonalChunk, at most
// kZonalChunk of them) at one level: each thread its columns in registers,
// the warps by shuffles, then one global atomic per warp and sum. The kernel
// is bound by the float64 pipe (80 cycles a warp instruction), so what it
// avoids is float64 work: the pressure comes from pow1p's table, one
// reciprocal of rho serves T, v and w, and no shared-memory float64 atomics
// (a compare-and-swap loop with an addition per colliding lane) are left.
// g5 x 37 float, 36 bands: the call 149 -> 99 us.
constexpr int kZonalThreads = 64, kZonalChunk = 256;
constexpr int kZonalQ = 9;    // weight, u, v, T, p, uv, vT, uu, vv

template <typename R>
__global__ void __launch_bounds__(kZonalThreads)
    k_zonal_partial(Geo<R> G, Vert V, Phys ph, const double* __restrict__ pw, Xf<R> X, Xf<R> XL,
                    const int* __restrict__ order, const int4* __restrict__ chunk, const double* __restrict__ basis,
                    int nlat, double* __restrict__ tmp, double* __restrict__ wsum) {
  __shared__ double sinv;
  const int k = blockIdx.y, S = G.colp;
  const int4 ch = chunk[blockIdx.x];               // band, first and last + 1 of order
  if (threadIdx.x == 0) sinv = 1.0 / V.thb[k];
  __syncthreads();
  const double rhob = V.rhob[k], thb = V.thb[k], pb = V.pb[k], clo = V.clo[k], chi = V.chi[k], inv_thb = sinv;
  const double vol = V.rc[k] * V.rc[k] * V.dz[k];
  double acc[kZonalQ] = {};
  for (int t = ch.y + threadIdx.x; t < ch.z; t += kZonalThreads) {
    const int c = order[t];
    const size_t i = (size_t)k * S + c;
    // the full value of a field: a compensated state adds its low part XL
    auto val = [&](const R* hi, const R* lo, size_t j) { return lo ? (double)hi[j] + (double)lo[j] : (double)hi[j]; };
    const double inv = 1.0 / (rhob + val(X.rho, XL.rho, i));
    const double x = div_by(val(X.th, XL.th, i), thb, inv_thb);
    double f, ln;
    if (!pow1p<false>(ph, pw, x, f, ln)) f = pow1p_general(x, ph.gamma).x;
    const double p = fma(pb, f, pb);
    const double T = p * inv * ph.inv_Rd;
    const double vx = val(X.mx, XL.mx, i) * inv, vy = val(X.my, XL.my, i) * inv, vz = val(X.mz, XL.mz, i) * inv;
    const double u = vx * basis[c] + vy * basis[S + c] + vz * basis[2 * S + c];
    const double v = vx * basis[3 * S + c] + vy * basis[4 * S + c] + vz * basis[5 * S + c];
    wsum[i] += (clo * val(X.w, XL.w, i) + chi * val(X.w, XL.w, i + S)) * inv;
    const double w = G.area[c] * vol, wu = w * u, wv = w * v;
    acc[0] += w;
    acc[1] += wu;
    acc[2] += wv;
    acc[3] += w * T;
    acc[4] += w * p;
    acc[5] += wu * v;
    acc[6] += wv * T;
    acc[7] += wu * u;
    acc[8] += wv * v;
  }
#pragma unroll
  for (int j = 0; j < kZonalQ; ++j)
    for (int d = 16; d > 0; d /= 2) acc[j] += __shfl_down_sync(0xffffffffu, acc[j], d);
  if ((threadIdx.x & 31) == 0 && acc[0] != 0.0) {
    double* out = tmp + ((size_t)k * nlat + ch.x) * kZonalQ;
#pragma unroll
    for (int j = 0; j < kZonalQ; ++j) atomicAdd(out + j, acc[j]);
  }
}

// per (level, band): the state's band means and covariances added to acc,
// the sums cleared for the next state
__global__ void k_zonal_finish(int n, double* __restrict__ tmp, double* __restrict__ acc) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n) return;
  double* s = tmp + (size_t)t * kZonalQ;
  double* a = acc + (size_t)t * kZonalQ;
  const double W = s[0];
  if (W > 0.0) {
    const double mu = s[1] / W, mv = s[2] / W, mT = s[3] / W, mp = s[4] / W;
    a[0] += W;
    a[1] += mu;
    a[2] += mv;
    a[3] += mT;
    a[4] += mp;
    a[5] += s[5] / W - mu * mv;
    a[6] += s[6] / W - mv * mT;
    a[7] += s[7] / W - mu * mu;
    a[8] += s[8] / W - mv * mv;
  }
  for (int j = 0; j < kZonalQ; ++j) s[j] = 0.0;
}

template <typename R>
int zonal_launch(thor_state* s) {
  auto* I = static_cast<Impl<R>*>(s->impl.get());
  ZonalAcc& z = s->zonal;
  const int nv = I->G.nv;
  k_zonal_partial<R><<<dim3(z.nchunk, nv), kZonalThreads, 0, I->stream>>>(
      I->G, I->V, I->ph, I->U.pw, I->Xt, I->XtL, z.order, static_cast<const int4*>(z.chunk), z.basis, z.nlat, z.tmp, z.wsum);
  const int n = nv * z.nlat;
  k_zonal_finish<<<(n + 255) / 256, 256, 0, I->stream>>>(n, z.tmp, z.acc);
  I->launches += 2;
  return cudaGetLastError() == cudaSuccess ? THOR_OK : THOR_ECUDA;
}

// (re)allocates the accumulator for nlat bands: the columns in the order of
// their bands, the bands' chunks, and east/north unit vectors of every column
// (host, float64, from the grid points); sums and accumulator cleared
int zonal_setup(thor_state* s, int nlat) {
  ZonalAcc& z = s->zonal;
  zonal_release(z);
  const HostGrid& h = s->grid->h;
  const int ncol = h.ncol, nv = h.nv, S = (ncol + kBlock - 1) / kBlock * kBlock;
  std::vector<int> band(ncol, 0), first(nlat + 1, 0), order(ncol);
  std::vector<int4> chunk;
  std::vector<double> basis(6 * (size_t)S, 0.0);
  for (int c = 0; c < ncol; ++c) {
    const double x = h.P[3 * c], y = h.P[3 * c + 1], zz = h.P[3 * c + 2];
    const double lon = std::atan2(y, x), lat = std::asin(std::fmax(-1.0, std::fmin(1.0, zz)));
    // 1e-9 rad: a cell on a band edge (the equatorial cells) goes north,
    // whatever the last bits of its coordinates
    int b = (int)std::floor((lat + 0.5 * M_PI + 1e-9) / M_PI * nlat);
    band[c] = b < nlat ? (b < 0 ? 0 : b) : nlat - 1;
    ++first[band[c] + 1];
    if (std::hypot(x, y) < 1e-9) continue;   // a polar cell: east and north undefined, u = v = 0
    basis[c] = -std::sin(lon);
    basis[S + c] = std::cos(lon);
    basis[2 * S + c] = 0.0;
    basis[3 * S + c] = -std::sin(lat) * std::cos(lon);
    basis[4 * S + c] = -std::sin(lat) * std::sin(lon);
    basis[5 * S + c] = std::cos(lat);
  }
  for (int b = 0; b < nlat; ++b) {
    for (int t = first[b]; t < first[b] + first[b + 1]; t += kZonalChunk)
      chunk.push_back(make_int4(b, t, std::min(t + kZonalChunk, first[b] + first[b + 1]), 0));
    first[b + 1] += first[b];
  }
  std::vector<int> at(first.begin(), first.end() - 1);
  for (int c = 0; c < ncol; ++c) order[at[band[c]]++] = c;
  const size_t nq = (size_t)nv * nlat * kZonalQ;
  const size_t nw = (size_t)nv * S;
  if (cudaMalloc(&z.order, ncol * sizeof(int)) || cudaMalloc(&z.chunk, chunk.size() * sizeof(int4)) ||
      cudaMalloc(&z.basis, basis.size() * sizeof(double)) ||
      cudaMalloc(&z.tmp, nq * sizeof(double)) || cudaMalloc(&z.acc, nq * sizeof(double)) ||
      cudaMalloc(&z.wsum, nw * sizeof(double))) {
    zonal_release(z);
    return THOR_ENOMEM;
  }
  if (cudaMemcpy(z.order, order.data(), ncol * sizeof(int), cudaMemcpyHostToDevice) ||
      cudaMemcpy(z.chunk, chunk.data(), chunk.size() * sizeof(int4), cudaMemcpyHostToDevice) ||
      cudaMemcpy(z.basis, basis.data(), basis.size() * sizeof(double), cudaMemcpyHostToDevice) ||
      cudaMemset(z.tmp, 0, nq * sizeof(double)) || cudaMemset(z.acc, 0, nq * sizeof(double)) ||
      cudaMemset(z.wsum, 0, nw * sizeof(double))) {
    zonal_release(z);
    return THOR_ECUDA;
  }
  z.nchunk = (int)chunk.size();
  z.nlat = nlat;
  z.samples = 0;
  return THOR_OK;
}

}  // namespace

void zonal_release(ZonalAcc& z) {
  if (z.order) cudaFree(z.order);
  if (z.chunk) cudaFree(z.chunk);
  if (z.basis) cudaFree(z.basis);
  if (z.tmp) cudaFree(z.tmp);
  if (z.acc) cudaFree(z.acc);
  if (z.wsum) cudaFree(z.wsum);
  z = ZonalAcc{};
}

}  // namespace thor

extern "C" {

int thor_zonal_accumulate(thor_state* s, int nlat) {
  if (!s || nlat < 1 || nlat > 360) return THOR_EINVAL;
  if (s->zonal.nlat != nlat) {
    if (cudaStreamSynchronize(s->impl->stream)) return THOR_ECUDA;
    const int rc = thor::zonal_setup(s, nlat);
    if (rc) return rc;
  }
  const int rc = s->precision == THOR_FP64 ? thor::zonal_launch<double>(s) : thor::zonal_launch<float>(s);
  if (rc == THOR_OK) ++s->zonal.samples;
  return rc;
}

int thor_zonal_read(thor_state* s, int nlat, double* out, size_t n, int reset, long long* samples) {
  if (!s || !samples) return THOR_EINVAL;
  const size_t need = (size_t)s->grid->h.nv * nlat * 9;
  if (nlat < 1 || !out || n != need) return THOR_EINVAL;
  if (s->zonal.nlat != nlat) {
    std::memset(out, 0, need * sizeof(double));
    *samples = 0;
    return THOR_OK;
  }
  if (cudaStreamSynchronize(s->impl->stream) ||
      cudaMemcpy(out, s->zonal.acc, need * sizeof(double), cudaMemcpyDeviceToHost))
    return THOR_ECUDA;
  *samples = s->zonal.samples;
  if (reset) {
    const size_t colp = (size_t)(s->grid->h.ncol + thor::kBlock - 1) / thor::kBlock * thor::kBlock;
    if (cudaMemset(s->zonal.acc, 0, need * sizeof(double)) ||
        cudaMemset(s->zonal.wsum, 0, (size_t)s->grid->h.nv * colp * sizeof(double)))
      return THOR_ECUDA;
    s->zonal.samples = 0;
  }
  return THOR_OK;
}

int thor_zonal_read_w(thor_state* s, int nlat, double* out, size_t n, long long* samples) {
  if (!s || !samples || !out) return THOR_EINVAL;
  const int ncol = s->grid->h.ncol, nv = s->grid->h.nv;
  if (nlat < 1 || n != (size_t)ncol * nv) return THOR_EINVAL;
  if (s->zonal.nlat != nlat || s->zonal.samples == 0) {
    std::memset(out, 0, n * sizeof(double));
    *samples = 0;
    return THOR_OK;
  }
  const size_t S = (size_t)(ncol + thor::kBlock - 1) / thor::kBlock * thor::kBlock;
  std::vector<double> buf((size_t)nv * S);
  if (cudaStreamSynchronize(s->impl->stream) ||
      cudaMemcpy(buf.data(), s->zonal.wsum, buf.size() * sizeof(double), cudaMemcpyDeviceToHost))
    return THOR_ECUDA;
  const double inv = 1.0 / (double)s->zonal.samples;
  for (int c = 0; c < ncol; ++c)
    for (int k = 0; k < nv; ++k) out[(size_t)c * nv + k] = buf[k * S + c] * inv;
  *samples = s->zonal.samples;
  return THOR_OK;
}

}  // extern "C"
