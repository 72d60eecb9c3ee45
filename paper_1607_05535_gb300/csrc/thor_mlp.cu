// Learned per-column closure (an extension: the paper has no learned part).
//
// A dense MLP y = W_L^T relu(... relu(W_1^T x + b_1) ...) + b_L with float32
// master weights, bfloat16 weights and layer inputs on the tensor cores and
// float32 accumulation; trained with a mean-squared-error loss and Adam
// (Kingma and Ba 2015). The GEMMs run on the fifth-generation tensor cores:
// tcgen05.mma kind::f16 with bfloat16 operands in shared memory and the
// float32 accumulator in tensor memory, the operands brought in by TMA in
// the 128-byte swizzled layout (k_gemm_tma; transposed copies of the
// weights, layer inputs and gradients make every product read both operands
// along its contraction) or, without a tensor-map encoder, staged
// by threads (k_gemm_tc); the warp-level mma.sync m16n8k16 kernel
// (k_gemm_bf16) is kept as a switchable reference path (thor_mlp_tune).
//
// Closure: per column, the inputs are 5 fields (rho', M_x, M_y, M_z, Th') at
// all levels and the neighbour means of the same (as anomalies); the
// outputs are correction tendencies of the same 5 fields at all levels,
// added as field += dt * tendency after every large step. Training data come
// from high-resolution runs area-averaged onto the coarse grid
// (thor_coarse_grain).
#include <cuda.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <memory>
#include <mutex>
#include <new>
#include <utility>
#include <vector>

#include "../../include/thor.h"
#include "thor_state.h"

namespace thor {
namespace {

constexpr int BM = 64, BN = 64, BK = 16;   // block tile, 4 warps of 32 x 32

__device__ __forceinline__ uint32_t pack_bf16(__nv_bfloat16 lo, __nv_bfloat16 hi) {
  return (uint32_t)__bfloat16_as_ushort(lo) | ((uint32_t)__bfloat16_as_ushort(hi) << 16);
}

__device__ __forceinline__ void mma_bf16(float* d, const uint32_t* a, const uint32_t* b) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 "
      "{%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

// C[M][N] = op(A)[M][K] op(B)[K][N]; op(A)(m,k) = transA ? A[k*lda+m] : A[m*lda+k],
// op(B)(k,n) = transB ? B[n*ldb+k] : B[k*ldb+n]. Epilogue: + bias[n], relu,
// float32 store to C (ldc) and / or bfloat16 store to Cb (ldcb).
__global__ void __launch_bounds__(128) k_gemm_bf16(int M, int N, int K, const __nv_bfloat16* A, int lda,
                                                   int transA, const __nv_bfloat16* B, int ldb, int transB,
                                                   float* C, int ldc, const float* bias, int relu,
                                                   __nv_bfloat16* Cb, int ldcb) {
  __shared__ __align__(16) __nv_bfloat16 As[BM][BK + 8];
  __shared__ __align__(16) __nv_bfloat16 Bs[BK][BN + 8];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int g = lane >> 2, t = lane & 3;
  const int m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
  const int wm = (warp >> 1) * 32, wn = (warp & 1) * 32;
  const __nv_bfloat16 zero = __float2bfloat16(0.0f);
  float acc[2][4][4];
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int q = 0; q < 4; ++q) acc[i][j][q] = 0.0f;
  for (int k0 = 0; k0 < K; k0 += BK) {
    for (int e = tid; e < BM * BK; e += 128) {
      const int r = e / BK, kk = e % BK, m = m0 + r, k = k0 + kk;
      __nv_bfloat16 v = zero;
      if (m < M && k < K) v = transA ? A[(size_t)k * lda + m] : A[(size_t)m * lda + k];
      As[r][kk] = v;
    }
    for (int e = tid; e < BK * BN; e += 128) {
      const int kk = e / BN, c = e % BN, k = k0 + kk, n = n0 + c;
      __nv_bfloat16 v = zero;
      if (k < K && n < N) v = transB ? B[(size_t)n * ldb + k] : B[(size_t)k * ldb + n];
      Bs[kk][c] = v;
    }
    __syncthreads();
#pragma unroll
    for (int mi = 0; mi < 2; ++mi) {
      const int r = wm + mi * 16;
      uint32_t a[4];
      a[0] = pack_bf16(As[r + g][2 * t], As[r + g][2 * t + 1]);
      a[1] = pack_bf16(As[r + g + 8][2 * t], As[r + g + 8][2 * t + 1]);
      a[2] = pack_bf16(As[r + g][2 * t + 8], As[r + g][2 * t + 9]);
      a[3] = pack_bf16(As[r + g + 8][2 * t + 8], As[r + g + 8][2 * t + 9]);
#pragma unroll
      for (int ni = 0; ni < 4; ++ni) {
        const int c = wn + ni * 8;
        uint32_t b[2];
        b[0] = pack_bf16(Bs[2 * t][c + g], Bs[2 * t + 1][c + g]);
        b[1] = pack_bf16(Bs[2 * t + 8][c + g], Bs[2 * t + 9][c + g]);
        mma_bf16(acc[mi][ni], a, b);
      }
    }
    __syncthreads();
  }
#pragma unroll
  for (int mi = 0; mi < 2; ++mi)
#pragma unroll
    for (int ni = 0; ni < 4; ++ni)
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int m = m0 + wm + mi * 16 + g + (q >= 2 ? 8 : 0);
        const int n = n0 + wn + ni * 8 + 2 * t + (q & 1);
        if (m >= M || n >= N) continue;
        float v = acc[mi][ni][q];
        if (bias) v += bias[n];
        if (relu) v = v > 0.0f ? v : 0.0f;
        if (C) C[(size_t)m * ldc + n] = v;
        if (Cb) Cb[(size_t)m * ldcb + n] = __float2bfloat16(v);
      }
}

// g [m][N] <- g * (h > 0) (h rows of ldh), then gb = bf16(g) in rows of ldg
__global__ void k_relu_back(float* g, const __nv_bfloat16* h, int ldh, __nv_bfloat16* gb, int ldg, int m, int N,
                            int mask) {
  const size_t cnt = (size_t)m * N;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < cnt; i += (size_t)gridDim.x * blockDim.x) {
    const size_t r = i / N, n = i % N;
    float v = g[i];
    if (mask && !(__bfloat162float(h[r * ldh + n]) > 0.0f)) v = 0.0f;
    g[i] = v;
    gb[r * ldg + n] = __float2bfloat16(v);
  }
}

// column sums of g [M][N] in two deterministic passes: partial sums over
// row blocks of 128 (k_colsum_part: 32 columns x 8 row lanes per block,
// lanes added in a fixed order), then one warp per column adds the R
// partials part[R][N] in a fixed order (k_colsum_final)
__global__ void __launch_bounds__(256) k_colsum_part(const float* g, int M, int N, float* part) {
  __shared__ float s[8][33];
  const int tx = threadIdx.x, ty = threadIdx.y, n = blockIdx.x * 32 + tx, r0 = blockIdx.y * 128;
  const int r1 = min(r0 + 128, M);
  float a = 0.0f;
  if (n < N) {
#pragma unroll 4
    for (int r = r0 + ty; r < r1; r += 8) a += g[(size_t)r * N + n];
  }
  s[ty][tx] = a;
  __syncthreads();
  if (ty == 0 && n < N) {
    float t = 0.0f;
#pragma unroll
    for (int j = 0; j < 8; ++j) t += s[j][tx];
    part[(size_t)blockIdx.y * N + n] = t;
  }
}
__global__ void k_colsum_final(const float* part, int R, int N, float* out) {
  const int col = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
  if (col >= N) return;
  float t = 0.0f;
  for (int j = lane; j < R; j += 32) t += part[(size_t)j * N + col];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
  if (lane == 0) out[col] = t;
}

// dY = 2 (Y - T) / (M N); per-block partial sums of (Y - T)^2
__global__ void k_mse(const float* y, const float* t, float* dy, size_t n, float inv_n, float* part) {
  __shared__ float sh[256];
  float s = 0.0f;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    float d = y[i] - t[i];
    dy[i] = 2.0f * d * inv_n;
    s += d * d;
  }
  sh[threadIdx.x] = s;
  __syncthreads();
  for (int w = blockDim.x / 2; w > 0; w >>= 1) {
    if (threadIdx.x < w) sh[threadIdx.x] += sh[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) part[blockIdx.x] = sh[0];
}

// scale * (sum of part[0..n)), one block of 1024 threads, fixed-order tree
__global__ void __launch_bounds__(1024) k_sum_parts(const float* part, int n, float scale, float* out) {
  __shared__ float sh[1024];
  const int t = threadIdx.x;
  float a = 0.0f;
  for (int i = t; i < n; i += 1024) a += part[i];
  sh[t] = a;
  __syncthreads();
  for (int w = 512; w > 0; w >>= 1) {
    if (t < w) sh[t] += sh[t + w];
    __syncthreads();
  }
  if (t == 0) *out = sh[0] * scale;
}

// one Adam update of a float32 master weight
struct Adam {
  float lr, b1, b2, c1, c2, eps;
};
__device__ __forceinline__ float adam_step(const Adam& A, float p, float g, float& m, float& v) {
  m = A.b1 * m + (1.0f - A.b1) * g;
  v = A.b2 * v + (1.0f - A.b2) * g * g;
  return p - A.lr * (m / A.c1) / (sqrtf(v / A.c2) + A.eps);
}
__global__ void k_adam(float* p, const float* g, float* m, float* v, size_t n, Adam A) {
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    p[i] = adam_step(A, p[i], g[i], m[i], v[i]);
  }
}

inline int blocks_for(size_t n) { return (int)std::min<size_t>((n + 255) / 256, 4096); }

uint64_t splitmix(uint64_t x) {
  uint64_t z = x + 0x9E3779B97F4A7C15ULL;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
  return z ^ (z >> 31);
}


// ------------------------------------------------------------ tcgen05 GEMM
//
// One CTA of 4 warps computes a 128 x NT tile of C (NT <= 256, a multiple of
// 16): row r of the tile is tensor-memory lane r, column n is tensor-memory
// column n of a float32 accumulator. Per chunk of 64 k, all threads stage the
// bfloat16 operand tiles (128 x 64 of op(A), NT x 64 of op(B)^T) into shared
// memory in the canonical K-major layout without swizzle: 8 x 8 core
// matrices of 16-byte rows, core matrices adjacent in k 128 B apart (leading
// byte offset), groups of 8 rows 1024 B apart (stride byte offset). One
// thread then issues four 128 x NT x 16 MMAs and commits them to an
// mbarrier, which every thread waits on (bounded) before the tiles are
// overwritten. The epilogue reads the accumulator with tcgen05.ld (warp w
// owns lanes 32w..32w+31), adds the bias, applies the ReLU and stores.

constexpr int TC_M = 128, TC_KC = 64;

__device__ __forceinline__ uint32_t tc_core_off(int r, int k) {
  return (uint32_t)((((r >> 3) * (TC_KC / 8) + (k >> 3)) << 7) + ((r & 7) << 4) + ((k & 7) << 1));
}

// shared-memory matrix descriptor: start address, leading and stride byte
// offsets (all >> 4), the fixed version bits 46-48 = 0b001, no swizzle
__device__ __forceinline__ uint64_t tc_smem_desc(uint32_t addr, uint32_t lbo, uint32_t sbo) {
  return (uint64_t)((addr & 0x3FFFFu) >> 4) | ((uint64_t)((lbo >> 4) & 0x3FFFu) << 16) |
         ((uint64_t)((sbo >> 4) & 0x3FFFu) << 32) | (1ull << 46);
}

// instruction descriptor of kind::f16: float32 D (bits 4-5 = 1), bfloat16 A
// and B (bits 7-9, 10-12 = 1), both K-major, N >> 3 at bit 17, M >> 4 at 24
__host__ __device__ constexpr uint32_t tc_idesc(int M, int N) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ void tc_alloc(uint32_t* dst, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(dst)), "r"(ncols)
               : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tc_dealloc(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tc_fence_before() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_mma(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d),
      "l"(a), "l"(b), "r"(idesc), "r"(accumulate)
      : "memory");
}
__device__ __forceinline__ void tc_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
               : "memory");
}
__device__ __forceinline__ void tc_ld16(uint32_t taddr, uint32_t* v) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, "
      "[%16];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]),
        "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
      : "r"(taddr)
      : "memory");
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

__host__ __device__ constexpr int tc_cols(int nt) { return nt <= 32 ? 32 : nt <= 64 ? 64 : nt <= 128 ? 128 : 256; }

// Stages rows [r0, r0 + R) x k [k0, k0 + 64) of op(X) into core-matrix order
// at dst; op(X)(r, k) = X[r * ld + k] if kcontig, else X[k * ld + r]; zero
// outside rows_total x K. vec: ld a multiple of 8 and X 16-byte aligned, so
// full 8-element groups move as 16-byte vectors (transposed in registers when
// the source runs along r).
__device__ __forceinline__ void tc_stage(unsigned char* dst, const __nv_bfloat16* X, int ld, bool kcontig, int r0,
                                         int R, int rows_total, int k0, int K, bool vec, int tid) {
  const unsigned short* Xs = reinterpret_cast<const unsigned short*>(X);
  auto at = [&](int r, int k) -> uint32_t {
    if (r >= rows_total || k >= K) return 0u;
    return kcontig ? Xs[(size_t)r * ld + k] : Xs[(size_t)k * ld + r];
  };
  if (kcontig) {
    for (int u = tid; u < R * 8; u += 128) {
      const int r = u >> 3, kg = u & 7, row = r0 + r, k = k0 + kg * 8;
      uint4 v = make_uint4(0u, 0u, 0u, 0u);
      if (row < rows_total) {
        if (vec && k + 8 <= K) {
          v = *reinterpret_cast<const uint4*>(Xs + (size_t)row * ld + k);
        } else {
          v.x = at(row, k) | (at(row, k + 1) << 16);
          v.y = at(row, k + 2) | (at(row, k + 3) << 16);
          v.z = at(row, k + 4) | (at(row, k + 5) << 16);
          v.w = at(row, k + 6) | (at(row, k + 7) << 16);
        }
      }
      *reinterpret_cast<uint4*>(dst + tc_core_off(r, kg * 8)) = v;
    }
  } else {
    const int G = R >> 3;
    for (int u = tid; u < G * 8; u += 128) {
      const int rg = u % G, kg = u / G, row = r0 + rg * 8, kb = k0 + kg * 8;
      uint32_t w[8][4];               // w[kk][j]: rows 2j, 2j+1 at k = kb + kk
      if (vec && row + 8 <= rows_total && kb + 8 <= K) {
#pragma unroll
        for (int kk = 0; kk < 8; ++kk) {
          const uint4 v = *reinterpret_cast<const uint4*>(Xs + (size_t)(kb + kk) * ld + row);
          w[kk][0] = v.x;
          w[kk][1] = v.y;
          w[kk][2] = v.z;
          w[kk][3] = v.w;
        }
      } else {
#pragma unroll
        for (int kk = 0; kk < 8; ++kk)
#pragma unroll
          for (int j = 0; j < 4; ++j) w[kk][j] = at(row + 2 * j, kb + kk) | (at(row + 2 * j + 1, kb + kk) << 16);
      }
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        uint4 lo, hi;                 // core rows 2j (low halves) and 2j + 1 (high halves), k = kb..kb+7
        lo.x = __byte_perm(w[0][j], w[1][j], 0x5410);
        lo.y = __byte_perm(w[2][j], w[3][j], 0x5410);
        lo.z = __byte_perm(w[4][j], w[5][j], 0x5410);
        lo.w = __byte_perm(w[6][j], w[7][j], 0x5410);
        hi.x = __byte_perm(w[0][j], w[1][j], 0x7632);
        hi.y = __byte_perm(w[2][j], w[3][j], 0x7632);
        hi.z = __byte_perm(w[4][j], w[5][j], 0x7632);
        hi.w = __byte_perm(w[6][j], w[7][j], 0x7632);
        *reinterpret_cast<uint4*>(dst + tc_core_off(rg * 8 + 2 * j, kg * 8)) = lo;
        *reinterpret_cast<uint4*>(dst + tc_core_off(rg * 8 + 2 * j + 1, kg * 8)) = hi;
      }
    }
  }
}

// same contract as k_gemm_bf16; NT = tile width; err: device flag set when
// an MMA completion is not seen within the wait bound. Two shared-memory
// stages: chunk c + 1 is staged while the MMAs of chunk c run.
__global__ void __launch_bounds__(128, 1) k_gemm_tc(int M, int N, int K, const __nv_bfloat16* A, int lda,
                                                    int transA, const __nv_bfloat16* B, int ldb, int transB,
                                                    float* C, int ldc, const float* bias, int relu,
                                                    __nv_bfloat16* Cb, int ldcb, int NT, int* err) {
  extern __shared__ __align__(1024) unsigned char tsm[];
  __shared__ uint64_t bar[2];
  __shared__ uint32_t tmem_base;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int m0 = blockIdx.y * TC_M, n0 = blockIdx.x * NT;
  const uint32_t ncols = (uint32_t)tc_cols(NT);
  const int stage_bytes = (TC_M + NT) * TC_KC * 2;
  const bool vecA = (lda % 8 == 0) && ((reinterpret_cast<uintptr_t>(A) & 15) == 0);
  const bool vecB = (ldb % 8 == 0) && ((reinterpret_cast<uintptr_t>(B) & 15) == 0);
  if (warp == 0) tc_alloc(&tmem_base, ncols);
  if (tid == 0) {
    mbar_init(&bar[0], 1);
    mbar_init(&bar[1], 1);
    mbar_init_fence();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_base;
  const uint32_t idesc = tc_idesc(TC_M, NT);
  const int nchunks = (K + TC_KC - 1) / TC_KC;
  uint32_t uses[2] = {0u, 0u};          // commits issued on each barrier
  bool ok = true;
  for (int c = 0; c < nchunks && ok; ++c) {
    const int b = c & 1;
    unsigned char* As = tsm + b * stage_bytes;
    unsigned char* Bs = As + TC_M * TC_KC * 2;
    if (c >= 2) ok = mbar_wait(&bar[b], (uses[b] - 1) & 1u);   // the MMAs that read this stage are done
    if (!__syncthreads_and(ok)) break;
    tc_stage(As, A, lda, !transA, m0, TC_M, M, c * TC_KC, K, vecA, tid);
    tc_stage(Bs, B, ldb, transB != 0, n0, NT, N, c * TC_KC, K, vecB, tid);
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // generic-proxy writes -> tensor cores
    __syncthreads();
    if (tid == 0) {
      tc_fence_after();
      const uint32_t a_addr = smem_u32(As), b_addr = smem_u32(Bs);
#pragma unroll
      for (int kk = 0; kk < TC_KC / 16; ++kk) {
        const uint64_t ad = tc_smem_desc(a_addr + kk * 256, 128, 1024);
        const uint64_t bd = tc_smem_desc(b_addr + kk * 256, 128, 1024);
        tc_mma(tmem, ad, bd, idesc, (c > 0 || kk > 0) ? 1u : 0u);
      }
      tc_commit(&bar[b]);
    }
    uses[b] += 1u;
  }
  // the last commit covers every MMA issued before it
  const int last = (nchunks - 1) & 1;
  if (ok) ok = __syncthreads_and(mbar_wait(&bar[last], (uses[last] - 1) & 1u));
  tc_fence_after();
  if (ok) {
    // 64-column slabs: tensor memory -> shared memory (row r at stride 65
    // floats), then coalesced rows to global memory
    float* slab = reinterpret_cast<float*>(tsm);
    for (int s0 = 0; s0 < NT; s0 += 64) {
      const int w = NT - s0 < 64 ? NT - s0 : 64;
      for (int c = 0; c < w; c += 16) {
        uint32_t v[16];
        tc_ld16(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)(s0 + c), v);
#pragma unroll
        for (int j = 0; j < 16; ++j) slab[(warp * 32 + lane) * 65 + c + j] = __uint_as_float(v[j]);
      }
      __syncthreads();
      for (int e = tid; e < TC_M * w; e += 128) {
        const int r = e / w, cc = e % w, row = m0 + r, n = n0 + s0 + cc;
        if (row < M && n < N) {
          float x = slab[r * 65 + cc];
          if (bias) x += bias[n];
          if (relu) x = x > 0.0f ? x : 0.0f;
          if (C) C[(size_t)row * ldc + n] = x;
          if (Cb) Cb[(size_t)row * ldcb + n] = __float2bfloat16(x);
        }
      }
      __syncthreads();
    }
  } else if (tid == 0) {
    atomicExch(err, 1);
    for (int q = 0; q < 2; ++q)          // bounded: let outstanding MMAs finish before freeing
      if (uses[q]) mbar_wait(&bar[q], (uses[q] - 1) & 1u);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) tc_dealloc(tmem, ncols);
}

// dynamic shared memory of k_gemm_tc: the two tiles, and enough on top that
// no more CTAs share an SM than its 512 tensor-memory columns can hold
size_t tc_smem_bytes(int nt) {
  const size_t tiles = 2 * (size_t)(TC_M + nt) * TC_KC * 2;
  const int ctas = 512 / tc_cols(nt);
  const size_t cap = (size_t)(228 * 1024) / ctas - 2048;
  return std::max(tiles, std::min(cap, (size_t)200 * 1024));
}

// ------------------------------------------------ TMA-fed tcgen05 GEMM
//
// C[M][N] = A B^T for operands that both run along k in global memory
// (A [M][lda], B [N][ldb], ld a multiple of 8 elements, 16-byte aligned).
// The copy engine brings 128 x 64 and NT x 64 bfloat16 boxes into shared
// memory in the 128-byte swizzled K-major layout: one 128-byte row per
// matrix row, its eight 16-byte chunks permuted by XOR with (row mod 8),
// groups of 8 rows 1024 B apart (the stride byte offset); the four MMAs of
// a 64-deep chunk start 32 B apart inside those rows. Rows and k outside
// the operands arrive as zeros (tensor-map bounds). Stages form a ring of
// S <= TMA_STAGES with a full barrier (copies landed, by transaction bytes) and
// an empty barrier (the MMAs that read the stage are done, by
// tcgen05.commit). One thread issues copies and MMAs; all four warps run
// the epilogue.
//
// At the closure's sizes (batch 1024, widths 160-320) a product takes 2-3 us
// and the network's step is bound by the number of dependent launches, so
// (1) the epilogue does the elementwise work of the pass it belongs to
// (GemmOut: bias, ReLU, the loss and its gradient, the ReLU mask of the
// backward pass, bfloat16 copies straight and transposed, column sums for the
// bias gradients), (2) one launch runs two independent products (the weight
// and the input gradient of a layer), and (3) the kernels of a pass are
// launched with programmatic stream serialization, each set up (barriers,
// tensor memory, descriptors) while the previous one drains. Training step of
// 320-256-256-256-160, 29 launches -> 10: at batch 1024 163 -> 71 us, at 64, 4096,
// 8192 and 10240 56, 101, 166 and 244 us (the host takes 21 us a step at each); forward and
// gradients of 370-256-256-256-185 at batch 1000, which the thread-staged kernel
// ran before the copies were padded: 510 -> 87 us (thor_mlp::aligned).

constexpr int TMA_STAGES = 4, TMA_KC = 64, kMaxSplit = 8;

// shared-memory matrix descriptor of the 128-byte swizzled K-major layout:
// stride byte offset 1024 (8-row atoms), leading byte offset unused within
// one swizzle row (encoded 1), version bits 46-47 = 1, layout type 2
// (SWIZZLE_128B) at bits 61-63
__device__ __forceinline__ uint64_t tc_desc_sw128(uint32_t addr) {
  return (uint64_t)((addr & 0x3FFFFu) >> 4) | (1ull << 16) | ((uint64_t)(1024 >> 4) << 32) | (1ull << 46) |
         (2ull << 61);
}

__device__ __forceinline__ void tma_load_box(uint32_t dst, const CUtensorMap* map, int x, int y, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::
          "r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(smem_u32(bar))
      : "memory");
}

// what the epilogue does with a product, in this order; null pointers: nothing
struct GemmOut {
  const float* bias;               // + bias[n]
  int relu;
  const float* target;             // result <- gscale (result - target), squares of the difference summed
  int ld_target;
  float gscale;
  float* loss;                     // [CTA of the job]
  const __nv_bfloat16* mask;       // result zeroed where mask <= 0 (rows of ldm, a multiple of 8)
  int ldm;
  float* C;                        // float32 rows of ldc; split z at C + z c_split
  int ldc;
  size_t c_split;
  __nv_bfloat16* Cb;               // bfloat16 rows of ldcb (a multiple of 8, at least N)
  int ldcb;
  __nv_bfloat16* CbT;              // bfloat16 transposed, rows of ldt
  int ldt;
  float* colsum;                   // [row tile][N] column sums
  int rows128;                     // its tiles: 32 rows (rows_colsum), or 128 (tile_colsum)
};
struct GemmJob {
  CUtensorMap a, b;
  int M, N, K, NT, stages, ntiles, mtiles, splits, kc_per;
  GemmOut o;
  int blocks() const { return ntiles * mtiles * splits; }
};
struct GemmPair {
  GemmJob j[2];
  int blocks0;                     // CTAs of the first job
};

// column sums over a warp's 32 rows (lane = row, 16 columns each) in rising
// row order, as the other column sums of the library run, through the warp's
// own piece of shared memory; lanes 0..15 return the sums. A tree of
// exchanged halves costs 16 shuffles instead (the training step 70.4 us, this
// way 70.9), but rounds differently, and Adam's first steps, which divide a
// gradient by its own size, carry such a difference into the weights.
__device__ __forceinline__ float rows_colsum(const float* x, float* sm, int lane) {
  __syncwarp();
#pragma unroll
  for (int j = 0; j < 16; ++j) sm[lane * 17 + j] = x[j];
  __syncwarp();
  float a = 0.0f;
  if (lane < 16) {
#pragma unroll
    for (int r = 0; r < 32; ++r) a += sm[r * 17 + lane];
  }
  return a;
}

// column sums over the tile's 128 rows in the order of k_colsum_part (eight
// strided row lanes, then the lanes); every thread of the block comes here,
// thread t < 16 returns column t's sum
__device__ __forceinline__ float tile_colsum(const float* x, float* sm, int tid) {
  float* lanes = sm + 128 * 17;
  __syncthreads();
#pragma unroll
  for (int j = 0; j < 16; ++j) sm[tid * 17 + j] = x[j];
  __syncthreads();
  const int col = tid & 15, ty = tid >> 4;
  float a = 0.0f;
#pragma unroll
  for (int r = 0; r < 16; ++r) a += sm[(ty + 8 * r) * 17 + col];
  lanes[ty * 17 + col] = a;
  __syncthreads();
  a = 0.0f;
  if (tid < 16) {
#pragma unroll
    for (int j = 0; j < 8; ++j) a += lanes[j * 17 + tid];
  }
  return a;
}

__global__ void __launch_bounds__(128, 1) k_gemm_tma(const __grid_constant__ GemmPair P, int* err) {
  extern __shared__ unsigned char tma_raw[];
  __shared__ uint64_t full[TMA_STAGES], empty[TMA_STAGES], done;   // the first S in use
  __shared__ uint32_t tmem_base;
  __shared__ int all_ok;
  __shared__ float wloss[4];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int which = (int)blockIdx.x >= P.blocks0 ? 1 : 0;
  const GemmJob& J = P.j[which];
  const GemmOut& O = J.o;
  const int bid = (int)blockIdx.x - which * P.blocks0;
  const int nt_id = bid % J.ntiles, mt_id = bid / J.ntiles % J.mtiles, z = bid / (J.ntiles * J.mtiles);
  const int M = J.M, N = J.N, K = J.K, NT = J.NT, S = J.stages;
  const int m0 = mt_id * TC_M, n0 = nt_id * NT;
  const uint32_t ncols = (uint32_t)tc_cols(NT);
  const uint32_t raw = smem_u32(tma_raw), base = (raw + 1023u) & ~1023u;   // swizzle atoms need 1024 B alignment
  const uint32_t a_bytes = TC_M * TMA_KC * 2, stage_bytes = (uint32_t)(TC_M + NT) * TMA_KC * 2;
  if (warp == 0) tc_alloc(&tmem_base, ncols);
  if (tid == 0) {
    for (int s = 0; s < S; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    mbar_init(&done, 1);
    mbar_init_fence();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  pdl_next();
  pdl_wait();
  const uint32_t tmem = tmem_base;
  // split-K: split z takes chunks [c0, c0 + nchunks) and stores its partial
  // product at C + z c_split
  const int c0 = z * J.kc_per;
  const int nchunks = min(J.kc_per, (K + TMA_KC - 1) / TMA_KC - c0);
  if (tid == 0) {
    const uint32_t idesc = tc_idesc(TC_M, NT);
    auto load = [&](int c) {
      const int s = c % S;
      const uint32_t a = base + (uint32_t)s * stage_bytes;
      mbar_arrive_expect_tx(&full[s], stage_bytes);
      tma_load_box(a, &J.a, (c0 + c) * TMA_KC, m0, &full[s]);
      tma_load_box(a + a_bytes, &J.b, (c0 + c) * TMA_KC, n0, &full[s]);
    };
    int issued = 0, c = 0;
    bool ok = true;
    for (; issued < nchunks && issued < S; ++issued) load(issued);
    for (; c < nchunks; ++c) {
      const int s = c % S;
      if (!mbar_wait(&full[s], (uint32_t)(c / S) & 1u)) {
        ok = false;
        break;
      }
      tc_fence_after();
      const uint32_t a = base + (uint32_t)s * stage_bytes, b = a + a_bytes;
#pragma unroll
      for (int kk = 0; kk < TMA_KC / 16; ++kk)
        tc_mma(tmem, tc_desc_sw128(a + kk * 32), tc_desc_sw128(b + kk * 32), idesc, (c > 0 || kk > 0) ? 1u : 0u);
      tc_commit(&empty[s]);
      // refill the stage of the previous chunk (issued == c - 1 + S)
      if (c >= 1 && issued < nchunks) {
        const int p = c - 1;
        if (!mbar_wait(&empty[p % S], (uint32_t)(p / S) & 1u)) {
          ok = false;
          ++c;
          break;
        }
        load(issued++);
      }
    }
    // on a timed-out wait, let the copies still in flight (chunks c .. issued - 1) land first (bounded)
    for (int q = c; q < issued; ++q) mbar_wait(&full[q % S], (uint32_t)(q / S) & 1u);
    tc_commit(&done);                                   // completes when every MMA issued above has
    const bool fin = mbar_wait(&done, 0u);
    all_ok = ok && fin;
    if (!(ok && fin)) atomicExch(err, 1);
  }
  __syncthreads();
  __syncwarp();
  tc_fence_after();
  if (all_ok) {
    // straight from the accumulator: lane r of warp w holds row 32w + r, 16
    // columns per tcgen05.ld; row-major stores move 16-byte vectors, the
    // transposed store is coalesced across the warp's 32 consecutive rows
    const int row = m0 + warp * 32 + lane;
    const bool live = row < M;
    float* C = O.C ? O.C + z * O.c_split : nullptr;
    const bool vec = C && O.ldc % 4 == 0 && (reinterpret_cast<uintptr_t>(C) & 15) == 0;
    float loss = 0.0f;
    for (int c = 0; c < NT; c += 16) {
      const int n = n0 + c;
      if (n >= N) break;                                 // warp-uniform
      uint32_t v[16];
      tc_ld16(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)c, v);
      const int left = min(16, N - n);
      float x[16];
#pragma unroll
      for (int j = 0; j < 16; ++j) {
        x[j] = __uint_as_float(v[j]);
        if (O.bias && j < left) x[j] += O.bias[n + j];
        if (O.relu) x[j] = x[j] > 0.0f ? x[j] : 0.0f;
      }
      if (O.target) {
        const float* t = O.target + (size_t)row * O.ld_target + n;
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          const float d = live && j < left ? x[j] - t[j] : 0.0f;
          loss += d * d;
          x[j] = O.gscale * d;
        }
      }
      if (O.mask) {
        const uint4* h = reinterpret_cast<const uint4*>(O.mask + (size_t)row * O.ldm + n);
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          const uint4 w = live && n + 8 * q < O.ldm ? h[q] : make_uint4(0u, 0u, 0u, 0u);
          const uint32_t u[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
          for (int j = 0; j < 8; ++j)
            if (!(__bfloat162float(__ushort_as_bfloat16((unsigned short)(u[j >> 1] >> (16 * (j & 1))))) > 0.0f))
              x[8 * q + j] = 0.0f;
        }
      }
      if (live) {
        if (C) {
          float* o = C + (size_t)row * O.ldc + n;
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            if (vec && 4 * q + 4 <= left) {
              *reinterpret_cast<float4*>(o + 4 * q) = make_float4(x[4 * q], x[4 * q + 1], x[4 * q + 2], x[4 * q + 3]);
            } else {
#pragma unroll
              for (int j = 4 * q; j < 4 * q + 4; ++j)
                if (j < left) o[j] = x[j];
            }
          }
        }
        if (O.Cb) {
          // columns beyond N are zero: they pad the row to a multiple of 8
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            if (8 * h >= left) break;
            const float* y = x + 8 * h;
            uint4 q;
            q.x = pack_bf16(__float2bfloat16(y[0]), __float2bfloat16(y[1]));
            q.y = pack_bf16(__float2bfloat16(y[2]), __float2bfloat16(y[3]));
            q.z = pack_bf16(__float2bfloat16(y[4]), __float2bfloat16(y[5]));
            q.w = pack_bf16(__float2bfloat16(y[6]), __float2bfloat16(y[7]));
            *reinterpret_cast<uint4*>(O.Cb + (size_t)row * O.ldcb + n + 8 * h) = q;
          }
        }
        if (O.CbT) {
#pragma unroll
          for (int j = 0; j < 16; ++j)
            if (j < left) O.CbT[(size_t)(n + j) * O.ldt + row] = __float2bfloat16(x[j]);
        }
      }
      if (O.colsum) {
        if (!live) {
#pragma unroll
          for (int j = 0; j < 16; ++j) x[j] = 0.0f;
        }
        // the ring's stages are free: every copy has landed and every MMA is done
        float* cs = reinterpret_cast<float*>(tma_raw + (base - raw));
        if (O.rows128) {
          const float t = tile_colsum(x, cs, tid);
          if (tid < min(left, 16)) O.colsum[(size_t)mt_id * N + n + tid] = t;
        } else {
          const float t = rows_colsum(x, cs + warp * 32 * 17, lane);
          if (lane < left && lane < 16 && m0 + warp * 32 < M) O.colsum[(size_t)(m0 / 32 + warp) * N + n + lane] = t;
        }
      }
    }
    if (O.loss) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) loss += __shfl_xor_sync(0xffffffffu, loss, o);
      if (lane == 0) wloss[warp] = loss;
      __syncthreads();
      if (tid == 0) O.loss[bid] = ((wloss[0] + wloss[1]) + wloss[2]) + wloss[3];
    }
  }
  tc_fence_before();
  __syncthreads();
  __syncwarp();
  if (warp == 0) tc_dealloc(tmem, ncols);
}

size_t tma_smem_bytes(int nt, int stages = TMA_STAGES) {
  return 1024 + (size_t)stages * (TC_M + nt) * TMA_KC * 2;
}

// x (float32 [m][K]) -> h (bfloat16 rows of ldh) and, unless null, its
// transpose hT ([K][ldt]) through a 32 x 32 shared-memory tile (both stores
// coalesced); with part the column sums of x over each row tile of the block,
// 32 rows (sub = 1, rising rows) or 128 (sub = 4, the order of
// k_colsum_part), in part[row tile][K]
__global__ void k_to_bf16_t(const float* x, __nv_bfloat16* h, int ldh, __nv_bfloat16* hT, int m, int K, int ldt,
                            float* part, int sub) {
  __shared__ float t[32][33];
  pdl_next();
  pdl_wait();
  const int k0 = blockIdx.x * 32, tx = threadIdx.x;
  float lane_sum = 0.0f;
  for (int s = 0; s < sub; ++s) {
    const int r0 = ((int)blockIdx.y * sub + s) * 32;
    if (s > 0) __syncthreads();
    for (int j = threadIdx.y; j < 32; j += 8) {
      const int r = r0 + j, k = k0 + tx;
      float v = 0.0f;
      if (r < m && k < K) {
        v = x[(size_t)r * K + k];
        h[(size_t)r * ldh + k] = __float2bfloat16(v);
      }
      t[j][tx] = v;
      lane_sum += v;
    }
    if (!hT && !part) continue;
    __syncthreads();
    if (hT) {
      for (int j = threadIdx.y; j < 32; j += 8) {
        const int k = k0 + j, r = r0 + tx;
        if (k < K && r < m) hT[(size_t)k * ldt + r] = __float2bfloat16(t[tx][j]);
      }
    }
  }
  if (!part) return;
  if (sub > 1) {
    __syncthreads();
    t[threadIdx.y][tx] = lane_sum;
    __syncthreads();
  }
  if (threadIdx.y == 0 && k0 + tx < K) {
    const int n = sub > 1 ? 8 : 32;
    float a = 0.0f;
#pragma unroll 8
    for (int j = 0; j < n; ++j) a += t[j][tx];
    part[(size_t)blockIdx.y * K + k0 + tx] = a;
  }
}

// The parameters of every layer in one launch. A block owns a 32 x 32 tile of
// one W_l, or eight biases of one b_l (a warp each). kGrad and kAdam add the
// split-K partials of dW_l and the row-tile partials of db_l in a fixed order;
// kAdam updates the master weights with them, kGrad stores them flat; kAdam
// and kCopy write the bfloat16 copies W_l (rows of Np) and W_l^T (rows of Kp)
// that the products read. With kAdam the last block sums the loss partials.
enum { kCopy = 0, kGrad = 1, kAdam = 2 };
struct ParamTable {
  int L;
  int K[15], N[15], Kp[15], Np[15], splits[15], blk0[16];     // blk0: first block of the layer; [L]: all
  unsigned long long woff[15], boff[15], wpoff[15], wtoff[15], wsoff[15], cpoff[15];
  int rtiles;                                                 // row tiles of the batch (column sums)
  int nloss;
  float loss_scale;
};
inline int weight_tiles(int K, int N) { return ((N + 31) / 32) * ((K + 31) / 32); }
template <int MODE>
__global__ void __launch_bounds__(256) k_params(float* p, float* am, float* av, const float* ws, const float* cpart,
                                                __nv_bfloat16* wp, __nv_bfloat16* wt, float* grad,
                                                const float* lpart, float* loss,
                                                const __grid_constant__ ParamTable T, Adam A) {
  __shared__ float t[32][33];
  const int tx = threadIdx.x, ty = threadIdx.y, b = blockIdx.x;
  pdl_next();
  pdl_wait();
  if (MODE == kAdam && b == T.blk0[T.L]) {
    float* sh = &t[0][0];
    const int q = ty * 32 + tx;
    float a = 0.0f;
    for (int i = q; i < T.nloss; i += 256) a += lpart[i];
    sh[q] = a;
    __syncthreads();
    for (int w = 128; w > 0; w >>= 1) {
      if (q < w) sh[q] += sh[q + w];
      __syncthreads();
    }
    if (q == 0 && loss) *loss = sh[0] * T.loss_scale;
    return;
  }
  int l = 0;
  while (b >= T.blk0[l + 1]) ++l;
  const int K = T.K[l], N = T.N[l], r = b - T.blk0[l], nw = ((N + 31) / 32) * ((K + 31) / 32);
  if (r >= nw) {
    const int n = (r - nw) * 8 + ty;
    if (MODE == kCopy || n >= N) return;
    const float* cp = cpart + T.cpoff[l];
    float g = 0.0f;
    for (int j = tx; j < T.rtiles; j += 32) g += cp[(size_t)j * N + n];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) g += __shfl_xor_sync(0xffffffffu, g, o);
    if (tx != 0) return;
    const size_t i = T.boff[l] + n;
    if (MODE == kAdam)
      p[i] = adam_step(A, p[i], g, am[i], av[i]);
    else
      grad[i] = g;
    return;
  }
  const int n0 = r % ((N + 31) / 32) * 32, k0 = r / ((N + 31) / 32) * 32, n = n0 + tx;
  for (int j = ty; j < 32; j += 8) {
    const int k = k0 + j;
    if (k >= K || n >= N) continue;
    const size_t i = T.woff[l] + (size_t)k * N + n;
    float v;
    if (MODE == kCopy) {
      v = p[i];
    } else {
      const float* w = ws + T.wsoff[l] + (size_t)k * T.Np[l] + n;
      const size_t plane = (size_t)K * T.Np[l];
      float g = w[0];
      for (int z = 1; z < T.splits[l]; ++z) g += w[z * plane];
      if (MODE == kGrad) {
        grad[i] = g;
        continue;
      }
      v = adam_step(A, p[i], g, am[i], av[i]);
      p[i] = v;
    }
    wp[T.wpoff[l] + (size_t)k * T.Np[l] + n] = __float2bfloat16(v);
    t[j][tx] = v;
  }
  if (MODE == kGrad) return;
  __syncthreads();
  for (int j = ty; j < 32; j += 8) {
    const int nn = n0 + j, k = k0 + tx;
    if (nn < N && k < K) wt[T.wtoff[l] + (size_t)nn * T.Kp[l] + k] = __float2bfloat16(t[tx][j]);
  }
}
}  // namespace
}  // namespace thor

// ================================================================== MLP

struct thor_mlp {
  std::vector<int> sizes;              // layer widths, n_layers + 1 entries
  std::vector<int> ps;                 // the same rounded up to multiples of 8: the rows of the bfloat16 copies
  int use_tc = 1;                      // tcgen05 TMA-fed (1) or thread-staged (2), mma.sync reference path (0)
  bool tma_ok = false;                 // the tensor-map encoder was found
  // Every width a multiple of 8. The sums over the batch of other networks
  // (dW_l, db_l) run in the order of the thread-staged path, dW_l unsplit, so
  // that a training run gives the same weights on either; forward and backward
  // of 370-256-256-256-185 at batch 1000: 64 us split, 87 us unsplit.
  bool aligned = true;
  bool fwd_tma = false;                // the last forward kept the transposed layer inputs
  int sms = 148;                       // streaming multiprocessors of the device
  int ldt = 0;                         // row length of the transposed buffers (max_batch rounded up to 64)
  int* err = nullptr;                  // device flag of the tcgen05 kernels
  int max_batch = 0;
  cudaStream_t stream = nullptr;
  size_t nparam = 0;
  std::vector<size_t> woff, boff;      // offsets of W_l and b_l in the flat parameter vector
  void* arena = nullptr;
  float *p = nullptr, *grad = nullptr, *m = nullptr, *v = nullptr;   // flat float32 [nparam]
  __nv_bfloat16* wp = nullptr;         // bf16 weights W_l [K][Np] at wpoff[l], zero beyond N
  __nv_bfloat16* wt = nullptr;         // bf16 transposed weights W_l^T [N][Kp] at wtoff[l], zero beyond K
  std::vector<size_t> wpoff, wtoff;
  std::vector<__nv_bfloat16*> h;       // layer inputs (bf16) [max_batch][ps[l]], zero beyond the width
  std::vector<__nv_bfloat16*> hT;      // their transposes [sizes[l]][ldt] (TMA-fed backward)
  __nv_bfloat16* gb[2] = {nullptr, nullptr};    // bf16 gradients [max_batch][max width], of a layer and the one below
  __nv_bfloat16* gbT[2] = {nullptr, nullptr};   // their transposes [max width][ldt]
  std::vector<float*> z;               // hidden outputs / gradients (float32) [max_batch][sizes[l+1]] (not TMA-fed)
  float* y = nullptr;                  // network output [max_batch][n_out] (not TMA-fed)
  float* dy = nullptr;                 // output gradient (not TMA-fed)
  float* part = nullptr;               // reduction partials
  float* cpart = nullptr;              // column-sum partials, [row tiles][sizes[l + 1]] at cpoff[l]
  float* ws = nullptr;                 // weight gradients, [splits][K][Np] at wsoff[l]
  std::vector<size_t> cpoff, wsoff, ws_splits;
  int last_m = 0;
  long long step_count = 0;
  // States that evaluate the network (thor_closure_attach). stream is that of
  // the last one attached; the others wait for updated, the event after the
  // last change of the weights, and a change waits for their reads.
  std::vector<std::shared_ptr<ClosureUse>> uses;
  cudaEvent_t updated = nullptr;
  std::mutex staged;                   // the batch buffers, lent to one state's evaluation at a time
  int n_layers() const { return (int)sizes.size() - 1; }
};

namespace thor {
namespace {

void gemm(const thor_mlp* net, int M, int N, int K, const __nv_bfloat16* A, int lda, int transA,
          const __nv_bfloat16* B, int ldb, int transB, float* C, int ldc, const float* bias, int relu,
          __nv_bfloat16* Cb, int ldcb) {
  cudaStream_t st = net->stream;
  if (net->use_tc) {
    // the widest tile (fewest re-stagings of A) that still gives about one
    // CTA per SM, else 64 columns
    const int mtiles = (M + TC_M - 1) / TC_M;
    int width = 64;
    for (int w : {256, 128})
      if (mtiles * ((N + w - 1) / w) >= 148) {
        width = w;
        break;
      }
    const int ntiles = (N + width - 1) / width;
    const int nt = ((N + ntiles - 1) / ntiles + 15) / 16 * 16;
    dim3 grid(ntiles, (M + TC_M - 1) / TC_M);
    k_gemm_tc<<<grid, 128, tc_smem_bytes(nt), st>>>(M, N, K, A, lda, transA, B, ldb, transB, C, ldc, bias, relu,
                                                    Cb, ldcb, nt, net->err);
    return;
  }
  dim3 grid((N + BN - 1) / BN, (M + BM - 1) / BM);
  k_gemm_bf16<<<grid, 128, 0, st>>>(M, N, K, A, lda, transA, B, ldb, transB, C, ldc, bias, relu, Cb, ldcb);
}

using EncodeTiled = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                 const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                 CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// looked up once; a second thread waits for the first one's answer
EncodeTiled encode_tiled() {
  static const EncodeTiled fn = []() -> EncodeTiled {
    void* f = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess)
      return nullptr;
    return reinterpret_cast<EncodeTiled>(f);
  }();
  return fn;
}

// tensor map of a bfloat16 operand X [rows][ld] read along k (k < kext):
// boxes of 64 k x box_rows rows, 128-byte swizzle, zeros outside
bool encode_operand(CUtensorMap* map, const __nv_bfloat16* X, int kext, int rows, int ld, int box_rows) {
  EncodeTiled enc = encode_tiled();
  if (!enc || (reinterpret_cast<uintptr_t>(X) & 15) || ld % 8) return false;
  const cuuint64_t dims[2] = {(cuuint64_t)kext, (cuuint64_t)rows};
  const cuuint64_t strides[1] = {(cuuint64_t)ld * 2};
  const cuuint32_t box[2] = {(cuuint32_t)TMA_KC, (cuuint32_t)box_rows};
  const cuuint32_t es[2] = {1, 1};
  return enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<__nv_bfloat16*>(X), dims, strides, box, es,
             CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Shape of one product on k_gemm_tma: the widest tile (fewest re-reads of A)
// that still gives a CTA per SM, else 16 columns; with split a long
// contraction on too few tiles (the weight gradients: K = batch) is split
// along k over the idle SMs into at most max_split partials
void gemm_shape(const thor_mlp* net, int M, int N, int K, bool split, int max_split, GemmJob& J) {
  J.M = M;
  J.N = N;
  J.K = K;
  J.mtiles = (M + TC_M - 1) / TC_M;
  int width = 16;
  for (int w : {256, 128, 64, 32})
    if (J.mtiles * ((N + w - 1) / w) >= net->sms) {
      width = w;
      break;
    }
  const int tiles = (N + width - 1) / width;
  J.NT = ((N + tiles - 1) / tiles + 15) / 16 * 16;
  J.ntiles = (N + J.NT - 1) / J.NT;
  const int nchunks = (K + TMA_KC - 1) / TMA_KC, ctas = J.mtiles * J.ntiles;
  J.splits = 1;
  if (split && 2 * ctas <= net->sms && nchunks >= 8)
    J.splits = std::min({(net->sms + ctas - 1) / ctas, nchunks / 4, max_split});
  J.kc_per = (nchunks + J.splits - 1) / J.splits;
  J.splits = (nchunks + J.kc_per - 1) / J.kc_per;
  J.o = GemmOut{};
}

bool gemm_operands(GemmJob& J, const __nv_bfloat16* A, int lda, const __nv_bfloat16* B, int ldb) {
  return encode_operand(&J.a, A, J.K, J.M, lda, TC_M) && encode_operand(&J.b, B, J.K, J.N, ldb, J.NT);
}

// a kernel of a pass, with programmatic serialization against the one before
template <typename... K, typename... V>
cudaError_t launch_pass(void (*kern)(K...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, V&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, std::forward<V>(args)...);
}

// one or two independent products in one launch
int gemm_launch(const thor_mlp* net, GemmPair& P, int jobs, cudaStream_t st) {
  P.blocks0 = P.j[0].blocks();
  const int total = P.blocks0 + (jobs > 1 ? P.j[1].blocks() : 0);
  // the deepest ring that still lets every CTA of the grid be resident at
  // once (a second, partial wave would double the time of a short product)
  const int per_sm = (total + net->sms - 1) / net->sms;
  int nt = P.j[0].NT;
  if (jobs > 1) nt = std::max(nt, P.j[1].NT);
  int stages = 2;
  for (int st = TMA_STAGES; st > 2; --st)
    if ((size_t)per_sm * (tma_smem_bytes(nt, st) + 2048) <= (size_t)227 * 1024 && per_sm * tc_cols(nt) <= 512) {
      stages = st;
      break;
    }
  for (int q = 0; q < jobs; ++q) P.j[q].stages = stages;
  return launch_pass(k_gemm_tma, total, 128, tma_smem_bytes(nt, stages), st, P, net->err) == cudaSuccess
             ? THOR_OK
             : THOR_ECUDA;
}

// row length in elements of the bfloat16 gradient buffers
int grad_ld(const thor_mlp* net, int l) { return net->ps[l + 1]; }

// forward for m rows of x (float32 [m][n_in] on the device) into y (float32
// [m][n_out]); train: instead of y, the gradient 2 (y - target) / (m n_out) of
// the mean-squared error into gb[0], gbT[0] and the column and loss partials
int mlp_forward_tma(thor_mlp* net, const float* x, int m, float* y, const float* target, int* nloss) {
  cudaStream_t st = net->stream;
  const int L = net->n_layers();
  dim3 g((net->sizes[0] + 31) / 32, (m + 31) / 32);
  if (launch_pass(k_to_bf16_t, g, dim3(32, 8), 0, st, x, net->h[0], net->ps[0], net->hT[0], m, net->sizes[0],
                  net->ldt, (float*)nullptr, 1))
    return THOR_ECUDA;
  for (int l = 0; l < L; ++l) {
    const int K = net->sizes[l], N = net->sizes[l + 1];
    const bool last = l + 1 == L;
    GemmPair P;
    GemmJob& J = P.j[0];
    gemm_shape(net, m, N, K, false, 1, J);
    // op(B) = W_l read along k from its transposed copy [N][Kp]
    if (!gemm_operands(J, net->h[l], net->ps[l], net->wt + net->wtoff[l], net->ps[l])) return THOR_ECUDA;
    J.o.bias = net->p + net->boff[l];
    if (!last) {
      J.o.relu = 1;
      J.o.Cb = net->h[l + 1];
      J.o.ldcb = net->ps[l + 1];
      J.o.CbT = net->hT[l + 1];
      J.o.ldt = net->ldt;
    } else if (target) {
      J.o.target = target;
      J.o.ld_target = N;
      J.o.gscale = 2.0f * (1.0f / ((float)m * (float)N));
      J.o.loss = net->part;
      J.o.Cb = net->gb[0];
      J.o.ldcb = grad_ld(net, l);
      J.o.CbT = net->gbT[0];
      J.o.ldt = net->ldt;
      J.o.colsum = net->cpart + net->cpoff[l];
      J.o.rows128 = !net->aligned;
      *nloss = J.blocks();
    } else {
      J.o.C = y;
      J.o.ldc = N;
    }
    int rc = gemm_launch(net, P, 1, st);
    if (rc) return rc;
  }
  net->fwd_tma = true;
  net->last_m = m;
  return THOR_OK;
}

// backward from the output gradient in gb[0], gbT[0] and its column partials:
// per layer one launch of dW_l = h_l^T g (into ws, both operands along the
// batch) and, above the first layer, g_{l-1} = (g W_l^T) masked by the ReLU
int mlp_backward_tma(thor_mlp* net, int m) {
  const int L = net->n_layers();
  for (int l = L - 1; l >= 0; --l) {
    const int K = net->sizes[l], N = net->sizes[l + 1], c = (L - 1 - l) & 1;
    GemmPair P;
    GemmJob &W = P.j[l > 0 ? 1 : 0], &X = P.j[0];
    gemm_shape(net, K, N, m, net->aligned, (int)net->ws_splits[l], W);
    if (!gemm_operands(W, net->hT[l], net->ldt, net->gbT[c], net->ldt)) return THOR_ECUDA;
    W.o.C = net->ws + net->wsoff[l];
    W.o.ldc = net->ps[l + 1];
    W.o.c_split = (size_t)K * net->ps[l + 1];
    if (l > 0) {
      // W_l [K][Np] runs along N, the contraction
      gemm_shape(net, m, K, N, false, 1, X);
      if (!gemm_operands(X, net->gb[c], grad_ld(net, l), net->wp + net->wpoff[l], net->ps[l + 1])) return THOR_ECUDA;
      X.o.mask = net->h[l];
      X.o.ldm = net->ps[l];
      X.o.Cb = net->gb[c ^ 1];
      X.o.ldcb = grad_ld(net, l - 1);
      X.o.CbT = net->gbT[c ^ 1];
      X.o.ldt = net->ldt;
      X.o.colsum = net->cpart + net->cpoff[l - 1];
      X.o.rows128 = !net->aligned;
    }
    int rc = gemm_launch(net, P, l > 0 ? 2 : 1, net->stream);
    if (rc) return rc;
  }
  return THOR_OK;
}

// k_params over every layer
template <int MODE>
int params_pass(const thor_mlp* net, int m, float* grad, int nloss, float loss_scale, float* loss, const Adam& A) {
  ParamTable T{};
  const int L = net->n_layers();
  T.L = L;
  T.rtiles = net->aligned ? (m + 31) / 32 : (m + 127) / 128;
  T.nloss = nloss;
  T.loss_scale = loss_scale;
  int b = 0;
  for (int l = 0; l < L; ++l) {
    const int K = net->sizes[l], N = net->sizes[l + 1];
    T.K[l] = K;
    T.N[l] = N;
    T.Kp[l] = net->ps[l];
    T.Np[l] = net->ps[l + 1];
    T.woff[l] = net->woff[l];
    T.boff[l] = net->boff[l];
    T.wpoff[l] = net->wpoff[l];
    T.wtoff[l] = net->wtoff[l];
    T.wsoff[l] = net->wsoff[l];
    T.cpoff[l] = net->cpoff[l];
    GemmJob J;
    gemm_shape(net, K, N, std::max(m, 1), net->aligned, (int)net->ws_splits[l], J);
    T.splits[l] = J.splits;
    T.blk0[l] = b;
    b += weight_tiles(K, N) + (N + 7) / 8;
  }
  T.blk0[L] = b;
  return launch_pass(k_params<MODE>, b + (MODE == kAdam ? 1 : 0), dim3(32, 8), 0, net->stream, net->p, net->m, net->v,
                     (const float*)net->ws, (const float*)net->cpart, net->wp, net->wt, grad,
                     (const float*)net->part, loss, T, A) == cudaSuccess
             ? THOR_OK
             : THOR_ECUDA;
}

// the bfloat16 copies of the weights from the master weights
int weights_copy(const thor_mlp* net) { return params_pass<kCopy>(net, 0, nullptr, 0, 0.0f, nullptr, Adam{}); }

bool tma_path(const thor_mlp* net) { return net->use_tc == 1 && net->tma_ok; }

// forward on the thread-staged tcgen05 or the mma.sync kernel, into net->y
int mlp_forward_staged(thor_mlp* net, const float* x, int m) {
  cudaStream_t st = net->stream;
  const int L = net->n_layers();
  net->fwd_tma = false;
  dim3 g((net->sizes[0] + 31) / 32, (m + 31) / 32);
  k_to_bf16_t<<<g, dim3(32, 8), 0, st>>>(x, net->h[0], net->ps[0], nullptr, m, net->sizes[0], 0, nullptr, 1);
  for (int l = 0; l < L; ++l) {
    const int K = net->sizes[l], N = net->sizes[l + 1];
    const float* b = net->p + net->boff[l];
    const __nv_bfloat16* W = net->wp + net->wpoff[l];
    if (l + 1 < L)
      gemm(net, m, N, K, net->h[l], net->ps[l], 0, W, net->ps[l + 1], 0, nullptr, 0, b, 1, net->h[l + 1], net->ps[l + 1]);
    else
      gemm(net, m, N, K, net->h[l], net->ps[l], 0, W, net->ps[l + 1], 0, net->y, N, b, 0, nullptr, 0);
  }
  net->last_m = m;
  return cudaGetLastError() == cudaSuccess ? THOR_OK : THOR_ECUDA;
}

// gradients of sum(y * dy) after a forward of the same batch into net->grad;
// dy float32 [m][n_out]
int mlp_backward_staged(thor_mlp* net, const float* dy, int m) {
  cudaStream_t st = net->stream;
  const int L = net->n_layers();
  // g (float32) lives in z[l] buffers: z[L-1] holds the output gradient
  float* g = net->z[L - 1];
  if (cudaMemcpyAsync(g, dy, (size_t)m * net->sizes[L] * sizeof(float), cudaMemcpyDeviceToDevice, st))
    return THOR_ECUDA;
  for (int l = L - 1; l >= 0; --l) {
    const int K = net->sizes[l], N = net->sizes[l + 1], ldg = grad_ld(net, l);
    float* gl = net->z[l];
    const __nv_bfloat16* W = net->wp + net->wpoff[l];
    // relu mask of this layer's output (hidden layers), then bf16 copy
    k_relu_back<<<blocks_for((size_t)m * N), 256, 0, st>>>(gl, l + 1 < L ? net->h[l + 1] : nullptr, net->ps[l + 1],
                                                           net->gb[0], ldg, m, N, l + 1 < L);
    // dW_l = h_l^T gb  ([K][N])
    gemm(net, K, N, m, net->h[l], net->ps[l], 1, net->gb[0], ldg, 0, net->grad + net->woff[l], N, nullptr, 0, nullptr, 0);
    // db_l = column sums of g
    k_colsum_part<<<dim3((N + 31) / 32, (m + 127) / 128), dim3(32, 8), 0, st>>>(gl, m, N, net->cpart);
    k_colsum_final<<<(N * 32 + 255) / 256, 256, 0, st>>>(net->cpart, (m + 127) / 128, N, net->grad + net->boff[l]);
    // g_{l-1} = gb W_l^T ([m][K]) into z[l-1]
    if (l > 0) gemm(net, m, K, N, net->gb[0], ldg, 0, W, net->ps[l + 1], 1, net->z[l - 1], K, nullptr, 0, nullptr, 0);
  }
  return cudaGetLastError() == cudaSuccess ? THOR_OK : THOR_ECUDA;
}

// y = MLP(x) for any number of rows through two scratch buffers of m rows x
// the widest layer, without the network's own batch buffers (inference), on
// the caller's stream
int mlp_infer(const thor_mlp* net, int m, float* y, __nv_bfloat16* const buf[2], cudaStream_t st) {
  const int L = net->n_layers();
  for (int l = 0; l < L; ++l) {
    const int K = net->sizes[l], N = net->sizes[l + 1];
    GemmPair P;
    GemmJob& J = P.j[0];
    gemm_shape(net, m, N, K, false, 1, J);
    if (!gemm_operands(J, buf[l & 1], net->ps[l], net->wt + net->wtoff[l], net->ps[l])) return THOR_ECUDA;
    J.o.bias = net->p + net->boff[l];
    if (l + 1 < L) {
      J.o.relu = 1;
      J.o.Cb = buf[(l & 1) ^ 1];
      J.o.ldcb = net->ps[l + 1];
    } else {
      J.o.C = y;
      J.o.ldc = N;
    }
    int rc = gemm_launch(net, P, 1, st);
    if (rc) return rc;
  }
  return THOR_OK;
}

// Around a change of the weights on net->stream: after the states that read
// them on other streams, and before their next evaluation. Nothing where the
// network serves one stream.
int weights_begin(const thor_mlp* net) {
  for (const std::shared_ptr<ClosureUse>& u : net->uses)
    if (u->stream != net->stream && cudaStreamWaitEvent(net->stream, u->read, 0)) return THOR_ECUDA;
  return THOR_OK;
}
int weights_end(const thor_mlp* net) {
  for (const std::shared_ptr<ClosureUse>& u : net->uses)
    if (u->stream != net->stream) return cudaEventRecord(net->updated, net->stream) ? THOR_ECUDA : THOR_OK;
  return THOR_OK;
}

}  // namespace
}  // namespace thor

extern "C" {

int thor_mlp_create(const int* sizes, int n_sizes, int max_batch, unsigned long long seed, void* stream,
                    thor_mlp** out) {
  using namespace thor;
  if (!sizes || !out || n_sizes < 2 || n_sizes > 16 || max_batch < 1) return THOR_EINVAL;
  for (int i = 0; i < n_sizes; ++i)
    if (sizes[i] < 1 || sizes[i] > 8192) return THOR_EINVAL;
  thor_mlp* net = new (std::nothrow) thor_mlp;
  if (!net) return THOR_ENOMEM;
  net->sizes.assign(sizes, sizes + n_sizes);
  net->max_batch = max_batch;
  net->stream = static_cast<cudaStream_t>(stream);
  const int L = n_sizes - 1;
  int wmax = 0;
  for (int l = 0; l < L; ++l) {
    net->woff.push_back(net->nparam);
    net->nparam += (size_t)sizes[l] * sizes[l + 1];
    net->boff.push_back(net->nparam);
    net->nparam += sizes[l + 1];
  }
  for (int i = 0; i < n_sizes; ++i) wmax = std::max(wmax, sizes[i]);
  // the TMA-fed products read rows of 16-byte multiples: the bfloat16 copies
  // of weights, layer inputs and gradients are padded with zeros to them
  net->tma_ok = encode_tiled() != nullptr;
  for (int i = 0; i < n_sizes; ++i) {
    net->ps.push_back((sizes[i] + 7) / 8 * 8);
    net->aligned = net->aligned && sizes[i] % 8 == 0;
  }
  net->ldt = (max_batch + 63) / 64 * 64;
  size_t nwp = 0, nwt = 0;
  for (int l = 0; l < L; ++l) {
    net->wpoff.push_back(nwp);
    nwp += ((size_t)sizes[l] * net->ps[l + 1] + 63) / 64 * 64;
    net->wtoff.push_back(nwt);
    nwt += ((size_t)sizes[l + 1] * net->ps[l] + 63) / 64 * 64;
  }
  {
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) == cudaSuccess &&
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess && sms > 0)
      net->sms = sms;
  }
  // one arena: params, grads, Adam moments, bf16 params, activations
  size_t bytes = 0;
  auto take = [&](size_t b) { size_t o = bytes; bytes += (b + 255) / 256 * 256; return o; };
  size_t o_p = take(net->nparam * 4), o_g = take(net->nparam * 4), o_m = take(net->nparam * 4),
         o_v = take(net->nparam * 4), o_wp = take(nwp * 2), o_wt = take(nwt * 2);
  const int wpad = (wmax + 7) / 8 * 8, rt = (max_batch + 31) / 32;
  std::vector<size_t> o_h, o_z, o_ht;
  for (int l = 0; l < L; ++l) o_h.push_back(take((size_t)max_batch * net->ps[l] * 2));
  for (int l = 0; l < L; ++l) o_z.push_back(take((size_t)max_batch * sizes[l + 1] * 4));
  size_t o_gb[2] = {0, 0}, o_gbt[2] = {0, 0};
  for (int q = 0; q < 2; ++q) o_gb[q] = take((size_t)max_batch * wpad * 2);
  // a loss partial per CTA of the output layer's product (at most 16 columns x 128 rows each)
  const size_t nparts = std::max<size_t>(4096, (size_t)((max_batch + TC_M - 1) / TC_M) * ((sizes[L] + 15) / 16));
  size_t o_y = take((size_t)max_batch * sizes[L] * 4), o_dy = take((size_t)max_batch * sizes[L] * 4),
         o_part = take(nparts * 4 + 64), o_err = take(64);
  size_t ncp = 0, nws = 0;
  for (int l = 0; l < L; ++l) {
    net->cpoff.push_back(ncp);
    ncp += (size_t)rt * sizes[l + 1];
    // room for the splits of the largest batch (a smaller one has no more)
    GemmJob J;
    gemm_shape(net, sizes[l], sizes[l + 1], max_batch, net->aligned, kMaxSplit, J);
    net->ws_splits.push_back(J.splits);
    net->wsoff.push_back(nws);
    nws += (size_t)J.splits * sizes[l] * net->ps[l + 1];
  }
  size_t o_cpart = take(ncp * 4), o_ws = take(nws * 4);
  for (int l = 0; l < L; ++l) o_ht.push_back(take((size_t)sizes[l] * net->ldt * 2));
  for (int q = 0; q < 2; ++q) o_gbt[q] = take((size_t)wmax * net->ldt * 2);
  if (cudaMalloc(&net->arena, bytes) != cudaSuccess) {
    delete net;
    return THOR_ENOMEM;
  }
  char* base = static_cast<char*>(net->arena);
  net->p = (float*)(base + o_p);
  net->grad = (float*)(base + o_g);
  net->m = (float*)(base + o_m);
  net->v = (float*)(base + o_v);
  net->wp = (__nv_bfloat16*)(base + o_wp);
  net->wt = (__nv_bfloat16*)(base + o_wt);
  for (int l = 0; l < L; ++l) {
    net->h.push_back((__nv_bfloat16*)(base + o_h[l]));
    net->z.push_back((float*)(base + o_z[l]));
    net->hT.push_back((__nv_bfloat16*)(base + o_ht[l]));
  }
  for (int q = 0; q < 2; ++q) {
    net->gb[q] = (__nv_bfloat16*)(base + o_gb[q]);
    net->gbT[q] = (__nv_bfloat16*)(base + o_gbt[q]);
  }
  net->y = (float*)(base + o_y);
  net->err = (int*)(base + o_err);
  net->ws = (float*)(base + o_ws);
  if (cudaMemsetAsync(net->err, 0, 64, net->stream) ||
      cudaFuncSetAttribute(k_gemm_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, 128 * 1024) ||
      cudaFuncSetAttribute(k_gemm_tma, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)tma_smem_bytes(256))) {
    cudaFree(net->arena);
    delete net;
    return THOR_ECUDA;
  }
  net->dy = (float*)(base + o_dy);
  net->part = (float*)(base + o_part);
  net->cpart = (float*)(base + o_cpart);
  // He-uniform initial weights from SplitMix64, zero biases
  std::vector<float> host(net->nparam, 0.0f);
  for (int l = 0; l < L; ++l) {
    const double a = std::sqrt(6.0 / sizes[l]);
    const size_t nw = (size_t)sizes[l] * sizes[l + 1];
    for (size_t i = 0; i < nw; ++i) {
      uint64_t r = splitmix(seed ^ (net->woff[l] + i));
      double u = (double)(r >> 11) * (1.0 / 9007199254740992.0);
      host[net->woff[l] + i] = (float)((2.0 * u - 1.0) * a);
    }
  }
  cudaStream_t st = net->stream;
  if (cudaMemsetAsync(net->arena, 0, bytes, st) ||
      cudaMemcpyAsync(net->p, host.data(), net->nparam * 4, cudaMemcpyHostToDevice, st)) {
    cudaFree(net->arena);
    delete net;
    return THOR_ECUDA;
  }
  if (weights_copy(net) || cudaStreamSynchronize(st)) {
    cudaFree(net->arena);
    delete net;
    return THOR_ECUDA;
  }
  *out = net;
  return THOR_OK;
}

int thor_mlp_info(const thor_mlp* net, size_t* nparam) {
  if (!net || !nparam) return THOR_EINVAL;
  *nparam = net->nparam;
  return THOR_OK;
}

int thor_mlp_get_params(thor_mlp* net, float* host, size_t n) {
  if (!net || !host || n != net->nparam) return THOR_EINVAL;
  int flag = 0;
  if (cudaMemcpyAsync(host, net->p, n * 4, cudaMemcpyDeviceToHost, net->stream)) return THOR_ECUDA;
  if (cudaMemcpyAsync(&flag, net->err, sizeof(int), cudaMemcpyDeviceToHost, net->stream)) return THOR_ECUDA;
  if (cudaStreamSynchronize(net->stream)) return THOR_ECUDA;
  return flag ? THOR_ETIMEOUT : THOR_OK;
}

int thor_mlp_tune(thor_mlp* net, int knob, int value) {
  if (!net) return THOR_EINVAL;
  if (knob == THOR_MLP_TUNE_TCGEN05) {
    if (value < 0 || value > 2) return THOR_EINVAL;
    net->use_tc = value;
    return THOR_OK;
  }
  return THOR_EINVAL;
}

int thor_mlp_set_params(thor_mlp* net, const float* host, size_t n) {
  using namespace thor;
  if (!net || !host || n != net->nparam) return THOR_EINVAL;
  if (weights_begin(net)) return THOR_ECUDA;
  if (cudaMemcpyAsync(net->p, host, n * 4, cudaMemcpyHostToDevice, net->stream)) return THOR_ECUDA;
  if (weights_copy(net)) return THOR_ECUDA;
  if (cudaMemsetAsync(net->m, 0, n * 4, net->stream) || cudaMemsetAsync(net->v, 0, n * 4, net->stream))
    return THOR_ECUDA;
  net->step_count = 0;
  return cudaStreamSynchronize(net->stream) ? THOR_ECUDA : THOR_OK;
}

int thor_mlp_forward(thor_mlp* net, const float* x, int m, float* y) {
  using namespace thor;
  if (!net || !x || !y || m < 1 || m > net->max_batch) return THOR_EINVAL;
  if (tma_path(net)) return mlp_forward_tma(net, x, m, y, nullptr, nullptr);
  int rc = mlp_forward_staged(net, x, m);
  if (rc) return rc;
  const size_t cnt = (size_t)m * net->sizes.back() * sizeof(float);
  return cudaMemcpyAsync(y, net->y, cnt, cudaMemcpyDeviceToDevice, net->stream) ? THOR_ECUDA : THOR_OK;
}

int thor_mlp_backward(thor_mlp* net, const float* dy, int m, float* grad) {
  using namespace thor;
  if (!net || !dy || !grad || m != net->last_m || m < 1) return THOR_EINVAL;
  // the TMA-fed products need the transposed inputs of a TMA-fed forward
  if (net->fwd_tma && tma_path(net)) {
    const int L = net->n_layers(), N = net->sizes[L], sub = net->aligned ? 1 : 4;
    dim3 g((N + 31) / 32, (m + 32 * sub - 1) / (32 * sub));
    if (launch_pass(k_to_bf16_t, g, dim3(32, 8), 0, net->stream, dy, net->gb[0], grad_ld(net, L - 1), net->gbT[0], m, N,
                    net->ldt, net->cpart + net->cpoff[L - 1], sub))
      return THOR_ECUDA;
    int rc = mlp_backward_tma(net, m);
    return rc ? rc : params_pass<kGrad>(net, m, grad, 0, 0.0f, nullptr, Adam{});
  }
  int rc = mlp_backward_staged(net, dy, m);
  if (rc) return rc;
  return cudaMemcpyAsync(grad, net->grad, net->nparam * 4, cudaMemcpyDeviceToDevice, net->stream) ? THOR_ECUDA
                                                                                              : THOR_OK;
}

int thor_mlp_train_step(thor_mlp* net, const float* x, const float* target, int m, float lr, float* loss) {
  using namespace thor;
  if (!net || !x || !target || m < 1 || m > net->max_batch || !(lr > 0)) return THOR_EINVAL;
  cudaStream_t st = net->stream;
  const size_t cnt = (size_t)m * net->sizes.back();
  auto adam = [&]() {
    net->step_count += 1;
    const float b1 = 0.9f, b2 = 0.999f;
    return Adam{lr, b1, b2, 1.0f - powf(b1, (float)net->step_count), 1.0f - powf(b2, (float)net->step_count), 1e-8f};
  };
  if (tma_path(net)) {
    int nloss = 0;
    int rc = mlp_forward_tma(net, x, m, nullptr, target, &nloss);
    if (!rc) rc = mlp_backward_tma(net, m);
    if (!rc) rc = weights_begin(net);
    if (!rc) rc = params_pass<kAdam>(net, m, nullptr, nloss, 1.0f / (float)cnt, loss, adam());
    return rc ? rc : weights_end(net);
  }
  int rc = mlp_forward_staged(net, x, m);
  if (rc) return rc;
  const int nb = std::min(blocks_for(cnt), 1024);
  k_mse<<<nb, 256, 0, st>>>(net->y, target, net->dy, cnt, 1.0f / (float)cnt, net->part);
  if (loss) k_sum_parts<<<1, 1024, 0, st>>>(net->part, nb, 1.0f / (float)cnt, loss);
  rc = mlp_backward_staged(net, net->dy, m);
  if (!rc) rc = weights_begin(net);
  if (rc) return rc;
  k_adam<<<blocks_for(net->nparam), 256, 0, st>>>(net->p, net->grad, net->m, net->v, net->nparam, adam());
  rc = weights_copy(net);
  if (!rc) rc = weights_end(net);
  if (rc) return rc;
  return cudaGetLastError() == cudaSuccess ? THOR_OK : THOR_ECUDA;
}

void thor_mlp_destroy(thor_mlp* net) {
  if (!net) return;
  if (net->arena) cudaFree(net->arena);
  if (net->updated) cudaEventDestroy(net->updated);
  delete net;
}

}  // extern "C"

// ================================================================ closure

namespace thor {
namespace {

constexpr int kClosureFields = 5;   // rho', M_x, M_y, M_z, Th'

template <typename R>
__device__ __forceinline__ const R* closure_field(const Xf<R>& X, int f) {
  return f == 0 ? X.rho : f == 1 ? X.mx : f == 2 ? X.my : f == 3 ? X.mz : X.th;
}
template <typename R>
__device__ __forceinline__ R* closure_field_rw(const Xf<R>& X, int f) {
  return f == 0 ? X.rho : f == 1 ? X.mx : f == 2 ? X.my : f == 3 ? X.mz : X.th;
}

// x[c][f nv + k] = field f at level k; x[c][5 nv + f nv + k] = the mean of
// that field over the neighbours of c minus its value at c (the neighbour
// anomaly carries the horizontal-curvature signal without the cancellation
// that bfloat16 inputs would suffer if centre and mean were given apart);
// normalised by (x - mean) / std per feature. Into float32 rows of F, or (Y =
// __nv_bfloat16) straight into the network's input rows of ldx.
//
// The planes run along the columns, the features along the levels: a block
// owns 32 columns x 32 levels of one field and turns them in shared memory,
// so that both sides move whole lines (one thread per column wrote every
// value to a line of its own). Sums over neighbours: float64 for
// float64 states; for float states the differences a(n) - a(c) as TwoSum
// pairs on the float32 pipes, about 48 bits, rounded once.
template <typename R>
struct NbrMean {
  R c, s = 0, e = 0;
  __device__ void add(R a);
  __device__ float anomaly(int nn) const;
};
template <>
__device__ __forceinline__ void NbrMean<double>::add(double a) { s += a; }
template <>
__device__ __forceinline__ float NbrMean<double>::anomaly(int nn) const { return (float)(s / nn - c); }
template <>
__device__ __forceinline__ void NbrMean<float>::add(float a) {
  float d, d1, t, t1;
  two_sum(a, -c, d, d1);
  two_sum(s, d, t, t1);
  s = t;
  e += d1 + t1;
}
template <>
__device__ __forceinline__ float NbrMean<float>::anomaly(int nn) const {
  // the quotient of s, corrected by its exact remainder and the low part: one rounding
  const float n = (float)nn, inv = 1.0f / n, q = s * inv;
  return q + (fmaf(-q, n, s) + e) * inv;
}
__device__ __forceinline__ void feature_store(float* x, float v) { *x = v; }
__device__ __forceinline__ void feature_store(__nv_bfloat16* x, float v) { *x = __float2bfloat16(v); }

template <typename R, typename Y>
__global__ void __launch_bounds__(256) k_features(Geo<R> G, Xf<R> X, const float* mean, const float* std, Y* x, int ldx) {
  __shared__ float tv[32][33], ta[32][33];
  const int S = G.colp, nv = G.nv, tx = threadIdx.x, ty = threadIdx.y;
  const int c0 = blockIdx.x * 32, c = c0 + tx, k0 = blockIdx.y * 32, f = blockIdx.z;
  if (c < G.ncol) {
    int nb[6], nn = 0;
#pragma unroll
    for (int j = 0; j < 6; ++j) {
      nb[j] = ld(G.nbr + j * S + c);
      nn += nb[j] != c;
    }
    for (int j = ty; j < 32 && k0 + j < nv; j += 8) {
      const R* a = closure_field(X, f) + (size_t)(k0 + j) * S;
      NbrMean<R> m{ld(a + c)};
#pragma unroll
      for (int q = 0; q < 6; ++q)
        if (nb[q] != c) m.add(ld(a + nb[q]));
      tv[j][tx] = (float)m.c;
      ta[j][tx] = m.anomaly(nn);
    }
  }
  __syncthreads();
  const int k = k0 + tx;
  if (k >= nv) return;
  const int j0 = f * nv + k, j1 = kClosureFields * nv + j0;
  const float m0 = mean[j0], s0 = std[j0], m1 = mean[j1], s1 = std[j1];
  for (int j = ty; j < 32 && c0 + j < G.ncol; j += 8) {
    Y* row = x + (size_t)(c0 + j) * ldx;
    feature_store(row + j0, (tv[tx][j] - m0) / s0);
    feature_store(row + j1, (ta[tx][j] - m1) / s1);
  }
}

// field += span (y * out_std + out_mean); the momentum correction is projected
// onto the tangent plane like every horizontal-momentum update. Blocks of 32
// columns x 32 levels, the network's rows turned in shared memory as above.
template <typename R>
__global__ void __launch_bounds__(256) k_apply(Geo<R> G, Xf<R> X, const float* y, const float* omean,
                                               const float* ostd, float span) {
  __shared__ float t[kClosureFields][32][33];
  const int S = G.colp, nv = G.nv, F = kClosureFields * nv, tx = threadIdx.x, ty = threadIdx.y;
  const int c0 = blockIdx.x * 32, k0 = blockIdx.y * 32;
  if (k0 + tx < nv) {
#pragma unroll
    for (int f = 0; f < kClosureFields; ++f) {
      const int q = f * nv + k0 + tx;
      const float sd = ostd[q], mn = omean[q];
      for (int j = ty; j < 32 && c0 + j < G.ncol; j += 8) t[f][j][tx] = y[(size_t)(c0 + j) * F + q] * sd + mn;
    }
  }
  __syncthreads();
  const int c = c0 + tx;
  if (c >= G.ncol) return;
  const float rx = (float)G.rhat[c], ry = (float)G.rhat[S + c], rz = (float)G.rhat[2 * S + c];
  for (int j = ty; j < 32 && k0 + j < nv; j += 8) {
    const size_t i = (size_t)(k0 + j) * S + c;
    float u[kClosureFields];
#pragma unroll
    for (int f = 0; f < kClosureFields; ++f) u[f] = t[f][tx][j];
    const float d = u[1] * rx + u[2] * ry + u[3] * rz;
    u[1] -= d * rx;
    u[2] -= d * ry;
    u[3] -= d * rz;
#pragma unroll
    for (int f = 0; f < kClosureFields; ++f) {
      R* a = closure_field_rw(X, f);
      a[i] = a[i] + (R)(span * u[f]);
    }
  }
}
template <typename R>
dim3 turn_grid(const Impl<R>* I, int fields) {
  return dim3((I->G.ncol + 31) / 32, (I->G.nv + 31) / 32, fields);
}

// tau_hat = MLP(features of the current state), kept in the binding's y buffer
template <typename R>
int closure_evaluate_t(thor_state* s) {
  Impl<R>* I = static_cast<Impl<R>*>(s->impl.get());
  ClosureBinding& cb = s->closure;
  thor_mlp* net = cb.net;
  cudaStream_t st = I->stream;
  const int ncol = I->G.ncol, nv = I->G.nv;
  const int Fin = 2 * kClosureFields * nv, Fout = kClosureFields * nv;
  const bool apart = net->stream != st;      // the network was attached to a state on another stream since
  if (tma_path(net)) {
    // features straight into the network's bfloat16 input rows, all columns
    // in one pass of the network through the binding's own buffers, the
    // output in place (10242 columns: 27 us; a pass of max_batch columns at a
    // time with float32 features and a copy of the output took about 390)
    k_features<R, __nv_bfloat16><<<turn_grid(I, kClosureFields), dim3(32, 8), 0, st>>>(
        I->G, I->Xt, cb.in_mean, cb.in_std, static_cast<__nv_bfloat16*>(cb.act[0]), net->ps[0]);
    __nv_bfloat16* const act[2] = {static_cast<__nv_bfloat16*>(cb.act[0]), static_cast<__nv_bfloat16*>(cb.act[1])};
    if (apart && cudaStreamWaitEvent(st, net->updated, 0)) return THOR_ECUDA;
    const int rc = mlp_infer(net, ncol, cb.y, act, st);
    if (rc) return rc;
    if (apart && cudaEventRecord(cb.use->read, st)) return THOR_ECUDA;
    I->launches += 1 + net->n_layers();
    return cudaGetLastError() == cudaSuccess ? THOR_OK : THOR_ECUDA;
  }
  k_features<R, float><<<turn_grid(I, kClosureFields), dim3(32, 8), 0, st>>>(I->G, I->Xt, cb.in_mean, cb.in_std, cb.x, Fin);
  // batches through the network's own buffers, hence on the network's stream
  std::lock_guard<std::mutex> lend(net->staged);
  if (apart && (cudaEventRecord(cb.use->read, st) || cudaStreamWaitEvent(net->stream, cb.use->read, 0))) return THOR_ECUDA;
  for (int c0 = 0; c0 < ncol; c0 += net->max_batch) {
    const int m = std::min(net->max_batch, ncol - c0);
    int rc = mlp_forward_staged(net, cb.x + (size_t)c0 * Fin, m);
    if (rc) return rc;
    if (cudaMemcpyAsync(cb.y + (size_t)c0 * Fout, net->y, (size_t)m * Fout * 4, cudaMemcpyDeviceToDevice, net->stream))
      return THOR_ECUDA;
  }
  if (apart && (cudaEventRecord(net->updated, net->stream) || cudaStreamWaitEvent(st, net->updated, 0))) return THOR_ECUDA;
  I->launches += 1 + (1 + net->n_layers()) * ((ncol + net->max_batch - 1) / net->max_batch);
  return cudaGetLastError() == cudaSuccess ? THOR_OK : THOR_ECUDA;
}

template <typename R>
int closure_correct_t(thor_state* s, double span) {
  Impl<R>* I = static_cast<Impl<R>*>(s->impl.get());
  ClosureBinding& cb = s->closure;
  k_apply<R><<<turn_grid(I, 1), dim3(32, 8), 0, I->stream>>>(I->G, I->Xt, cb.y, cb.out_mean, cb.out_std, (float)span);
  I->launches += 1;
  return cudaGetLastError() == cudaSuccess ? THOR_OK : THOR_ECUDA;
}

// One large step with the closure. The network sees the state at the start
// of each window of `period` large steps and its correction, period * dt *
// tau_hat, is added when the window closes: the coarse solution after n
// steps plus n dt tau, which is how the training target is defined.
template <typename R>
int closure_large_step_t(thor_state* s, int n_small, double dt) {
  ClosureBinding& cb = s->closure;
  int rc = THOR_OK;
  if (cb.counter % cb.period == 0) rc = closure_evaluate_t<R>(s);
  if (!rc) rc = s->impl->step(1, n_small, dt);
  if (rc) return rc;
  cb.counter += 1;
  if (cb.counter % cb.period == 0) rc = closure_correct_t<R>(s, cb.period * dt);
  return rc;
}

// Coarse graining. The caller's map (one coarse column per fine column, in
// host memory) is uploaded and turned into member lists on the device: the
// members of a coarse column are counted, each column takes a segment of the
// list (in any order: only the order within a segment enters the sums), the
// segments are filled, and sorted by rank so that every sum runs over rising
// fine columns whatever the atomics' order. kCgBad is set for an index out of
// range or a coarse column without members, kCgLong for a column with more
// than kCgRank members (ranking compares every member with every other); the
// kernels that follow then do nothing, so a refused map costs no more than its
// count, and lists with a long segment are built on the host in one pass over the
// map and averaged in a second launch. Building all lists on the host, with three
// buffers allocated and freed around it, made the call 260 us at g6 -> g5 x 32;
// now it is 121 us: 12 us for the map's upload, 20 us for the lists, 67 us for
// the averages (bound by the float64 pipe, 82% busy: building the doubles on
// the integer ALU instead of converting gave 68 us) and the read-back.
// The limit lies between the lengths measured on both sides, g6 x 32 onto
// coarser grids: longest list 267, 316 us on the device and 411 with the lists
// from the host; 995, 1292 and 986; 3426, 7050 and 2450.
constexpr int kCgRank = 512, kCgBad = 1, kCgLong = 2;
struct CoarseLists {
  int *map, *count, *start, *cursor, *raw, *member, *state;   // state[0] kCgBad | kCgLong, state[1] list length
  double* weight;
};

__global__ void k_cg_count(const int* __restrict__ map, int nfine, int ncol, int* count, int* state) {
  const int f = blockIdx.x * blockDim.x + threadIdx.x;
  if (f >= nfine) return;
  const int c = map[f];
  if (c < 0 || c >= ncol)
    atomicOr(state, kCgBad);
  else
    atomicAdd(count + c, 1);
}

// one warp's columns take one stretch of the list, with one atomic
__global__ void k_cg_start(const int* __restrict__ count, int ncol, int* start, int* cursor, int* state) {
  const int c = blockIdx.x * blockDim.x + threadIdx.x, lane = threadIdx.x & 31;
  const int n = c < ncol ? count[c] : 0;
  int sum = n;
  for (int d = 1; d < 32; d *= 2) {
    const int v = __shfl_up_sync(0xffffffffu, sum, d);
    if (lane >= d) sum += v;
  }
  int base = 0;
  if (lane == 31) base = atomicAdd(state + 1, sum);
  base = __shfl_sync(0xffffffffu, base, 31);
  if (c >= ncol) return;
  start[c] = cursor[c] = base + sum - n;
  if (n == 0) atomicOr(state, kCgBad);
  if (n > kCgRank) atomicOr(state, kCgLong);
}

__global__ void k_cg_fill(const int* __restrict__ map, int nfine, int ncol, const int* __restrict__ state, int* cursor,
                          int* raw) {
  const int f = blockIdx.x * blockDim.x + threadIdx.x;
  if (f >= nfine || state[0]) return;
  const int c = map[f];
  if (c >= 0 && c < ncol) raw[atomicAdd(cursor + c, 1)] = f;
}

// a warp per coarse column: members in rising order, and their weights
__global__ void k_cg_sort(const int* __restrict__ count, const int* __restrict__ start, int ncol,
                          const int* __restrict__ state, const int* __restrict__ raw, const double* __restrict__ area, int* member, double* weight) {
  const int c = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (c >= ncol || state[0]) return;
  const int n = count[c], s = start[c];
  for (int i = lane; i < n; i += 32) {
    const int f = raw[s + i];
    int rank = 0;
#pragma unroll 4
    for (int q = 0; q < n; ++q) rank += raw[s + q] < f;
    member[s + rank] = f;
    weight[s + rank] = area[f];
  }
  __syncwarp();
  double sum = 0.0;
#pragma unroll 4
  for (int q = 0; q < n; ++q) sum += weight[s + q];
  __syncwarp();
  for (int i = lane; i < n; i += 32) weight[s + i] /= sum;
}

// fine -> coarse area-weighted averages, the sums in float64; the low parts of
// a compensated coarse state (XcL) restart at zero
template <typename R>
__global__ void k_coarse_grain(Geo<R> Gc, Xf<R> Xf_, int Sf, Xf<R> Xc, Xf<R> XcL, CoarseLists L) {
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  const int k = blockIdx.y;               // 0..nv (interfaces use all nv+1)
  if (c >= Gc.ncol || L.state[0]) return;
  const int Sc = Gc.colp, nv = Gc.nv;
  double a[6] = {0, 0, 0, 0, 0, 0};
  const int e0 = L.start[c], e1 = e0 + L.count[c];
#pragma unroll 4
  for (int e = e0; e < e1; ++e) {
    const size_t i = (size_t)k * Sf + __ldg(L.member + e);
    const double w = __ldg(L.weight + e);
    if (k < nv) {
      a[0] += w * (double)Xf_.rho[i];
      a[1] += w * (double)Xf_.mx[i];
      a[2] += w * (double)Xf_.my[i];
      a[3] += w * (double)Xf_.mz[i];
      a[4] += w * (double)Xf_.th[i];
    }
    a[5] += w * (double)Xf_.w[i];
  }
  const size_t o = (size_t)k * Sc + c;
  if (k < nv) {
    const double rx = Gc.rhat[c], ry = Gc.rhat[Sc + c], rz = Gc.rhat[2 * Sc + c];
    const double d = a[1] * rx + a[2] * ry + a[3] * rz;
    Xc.rho[o] = (R)a[0];
    Xc.mx[o] = (R)(a[1] - d * rx);
    Xc.my[o] = (R)(a[2] - d * ry);
    Xc.mz[o] = (R)(a[3] - d * rz);
    Xc.th[o] = (R)a[4];
    if (XcL.rho) XcL.rho[o] = XcL.mx[o] = XcL.my[o] = XcL.mz[o] = XcL.th[o] = (R)0;
  }
  Xc.w[o] = (k == 0 || k == nv) ? (R)0 : (R)a[5];
  if (XcL.w) XcL.w[o] = (R)0;
}

}  // namespace

int closure_large_step(thor_state* s, int n_small, double dt) {
  return s->precision == THOR_FP64 ? closure_large_step_t<double>(s, n_small, dt)
                                   : closure_large_step_t<float>(s, n_small, dt);
}

void closure_release(thor_state* s) {
  if (s->closure.net) cudaStreamSynchronize(s->impl->stream);   // its last evaluation, before the network forgets it
  if (s->closure.y) cudaFree(s->closure.y);
  if (s->closure.act[0]) cudaFree(s->closure.act[0]);
  s->closure = ClosureBinding();
}

void coarse_release(CoarseWork& w) {
  if (w.buf) cudaFree(w.buf);
  if (w.ready) cudaEventDestroy(w.ready);
  w = CoarseWork();
}

}  // namespace thor

namespace {
template <typename R>
int features_t(thor_state* s, const float* mean, const float* std, float* x) {
  using namespace thor;
  Impl<R>* I = static_cast<Impl<R>*>(s->impl.get());
  k_features<R, float><<<turn_grid(I, kClosureFields), dim3(32, 8), 0, I->stream>>>(I->G, I->Xt, mean, std, x,
                                                                                 2 * kClosureFields * I->G.nv);
  I->launches += 1;
  return cudaGetLastError() == cudaSuccess ? THOR_OK : THOR_ECUDA;
}

template <typename R>
int coarse_t(thor_state* fine, thor_state* coarse, const int* map) {
  using namespace thor;
  Impl<R>* F = static_cast<Impl<R>*>(fine->impl.get());
  Impl<R>* C = static_cast<Impl<R>*>(coarse->impl.get());
  cudaStream_t st = C->stream;
  const int nf = F->G.ncol, nc = C->G.ncol;
  CoarseWork& w = coarse->coarse;
  // weight [nf], map, raw, member [nf], count [nc], state [2], start, cursor [nc]
  const size_t need = (size_t)nf * (sizeof(double) + 3 * sizeof(int)) + (3 * (size_t)nc + 2) * sizeof(int);
  if (w.bytes < need) {
    coarse_release(w);
    if (cudaMalloc(&w.buf, need)) {
      cudaGetLastError();
      w.buf = nullptr;
      return THOR_ENOMEM;
    }
    w.bytes = need;
  }
  if (!w.ready && cudaEventCreateWithFlags(&w.ready, cudaEventDisableTiming)) return THOR_ECUDA;
  CoarseLists L;
  L.weight = static_cast<double*>(w.buf);
  L.map = reinterpret_cast<int*>(L.weight + nf);
  L.raw = L.map + nf;
  L.member = L.raw + nf;
  L.count = L.member + nf;
  L.state = L.count + nc;
  L.start = L.state + 2;
  L.cursor = L.start + nc;
  auto average = [&]() {
    k_coarse_grain<R><<<dim3((nc + 127) / 128, C->G.nv + 1), 128, 0, st>>>(C->G, F->Xt, F->G.colp, C->Xt, C->XtL, L);
    return !cudaGetLastError();
  };
  bool ok = !cudaMemcpyAsync(L.map, map, nf * sizeof(int), cudaMemcpyHostToDevice, st) &&
            !cudaMemsetAsync(L.count, 0, ((size_t)nc + 2) * sizeof(int), st);
  // the fine state's tables and fields are complete on its own stream
  if (F->stream != st) ok = ok && !cudaEventRecord(w.ready, F->stream) && !cudaStreamWaitEvent(st, w.ready, 0);
  int state = 0;
  if (ok) {
    k_cg_count<<<(nf + 255) / 256, 256, 0, st>>>(L.map, nf, nc, L.count, L.state);
    k_cg_start<<<(nc + 255) / 256, 256, 0, st>>>(L.count, nc, L.start, L.cursor, L.state);
    k_cg_fill<<<(nf + 255) / 256, 256, 0, st>>>(L.map, nf, nc, L.state, L.cursor, L.raw);
    k_cg_sort<<<(nc + 7) / 8, 256, 0, st>>>(L.count, L.start, nc, L.state, L.raw, F->G.area, L.member, L.weight);
    ok = average() && !cudaMemcpyAsync(&state, L.state, sizeof(int), cudaMemcpyDeviceToHost, st);
    C->launches += 5;
  }
  // on every path: the map is the caller's, and the fine state may change after the call
  if (cudaStreamSynchronize(st) || !ok) return THOR_ECUDA;
  if (state & kCgBad) return THOR_EINVAL;
  if (!(state & kCgLong)) return THOR_OK;
  // the lists from the host: the same members in the same order
  std::vector<int> start(nc + 1, 0), count(nc), at(nc), member(nf);
  std::vector<double> area(nc, 0.0), weight(nf);
  for (int f = 0; f < nf; ++f) {
    ++start[map[f] + 1];
    area[map[f]] += fine->grid->h.area[f];
  }
  for (int c = 0; c < nc; ++c) {
    count[c] = start[c + 1];
    at[c] = start[c];
    start[c + 1] += start[c];
  }
  for (int f = 0; f < nf; ++f) {
    const int e = at[map[f]]++;
    member[e] = f;
    weight[e] = fine->grid->h.area[f] / area[map[f]];
  }
  ok = !cudaMemcpyAsync(L.start, start.data(), nc * sizeof(int), cudaMemcpyHostToDevice, st) &&
       !cudaMemcpyAsync(L.count, count.data(), nc * sizeof(int), cudaMemcpyHostToDevice, st) &&
       !cudaMemcpyAsync(L.member, member.data(), nf * sizeof(int), cudaMemcpyHostToDevice, st) &&
       !cudaMemcpyAsync(L.weight, weight.data(), nf * sizeof(double), cudaMemcpyHostToDevice, st) &&
       !cudaMemsetAsync(L.state, 0, sizeof(int), st) && average();
  if (ok) C->launches += 1;
  return cudaStreamSynchronize(st) || !ok ? THOR_ECUDA : THOR_OK;
}
}  // namespace

extern "C" {

int thor_closure_features(thor_state* s, const float* mean, const float* std, float* x) {
  if (!s || !mean || !std || !x) return THOR_EINVAL;
  return s->precision == THOR_FP64 ? features_t<double>(s, mean, std, x) : features_t<float>(s, mean, std, x);
}

int thor_closure_attach(thor_state* s, thor_mlp* net, const float* in_mean, const float* in_std,
                        const float* out_mean, const float* out_std, int period) {
  using namespace thor;
  if (!s) return THOR_EINVAL;
  closure_release(s);
  if (!net) return THOR_OK;                 // detached: plain method
  if (!in_mean || !in_std || !out_mean || !out_std || period < 1) return THOR_EINVAL;
  const int ncol = s->grid->h.ncol, nv = s->grid->h.nv;
  if (net->sizes.front() != 2 * kClosureFields * nv || net->sizes.back() != kClosureFields * nv)
    return THOR_EINVAL;
  ClosureBinding cb;
  cb.net = net;
  cb.in_mean = in_mean;
  cb.in_std = in_std;
  cb.out_mean = out_mean;
  cb.out_std = out_std;
  cb.period = period;
  // network buffers for every column: the output, and two of the widest layer
  // in bfloat16; the batched passes' float32 features lie over those two (they
  // take no more: an input row is 2 x 5 nv wide)
  int wmax = 0;
  for (int l = 0; l < net->n_layers(); ++l) wmax = std::max(wmax, net->ps[l]);
  const size_t act = (size_t)ncol * wmax * sizeof(__nv_bfloat16);
  const bool ok = !cudaMalloc(&cb.act[0], 2 * act) && !cudaMalloc(&cb.y, (size_t)ncol * kClosureFields * nv * 4);
  cb.act[1] = static_cast<char*>(cb.act[0]) + act;
  cb.x = static_cast<float*>(cb.act[0]);
  if (!ok) {
    s->closure = cb;
    closure_release(s);
    return THOR_ENOMEM;
  }
  // The network moves to the state's stream. What is queued on its old one
  // (training, another state's evaluation) comes first; that stream may be
  // gone by now, so the wait is for the device.
  cudaStream_t st = s->impl->stream;
  cb.use = std::make_shared<ClosureUse>();
  cb.use->stream = st;
  if ((net->stream != st && cudaDeviceSynchronize()) || cudaEventCreateWithFlags(&cb.use->read, cudaEventDisableTiming) ||
      (!net->updated && cudaEventCreateWithFlags(&net->updated, cudaEventDisableTiming))) {
    s->closure = cb;
    closure_release(s);
    return THOR_ECUDA;
  }
  net->uses.erase(std::remove_if(net->uses.begin(), net->uses.end(),
                                 [](const std::shared_ptr<ClosureUse>& u) { return u.use_count() == 1; }),
                  net->uses.end());
  net->uses.push_back(cb.use);
  net->stream = st;
  s->closure = cb;
  return THOR_OK;
}

int thor_coarse_grain(thor_state* fine, thor_state* coarse, const int* fine_to_coarse, size_t nfine) {
  if (!fine || !coarse || !fine_to_coarse || fine->precision != coarse->precision) return THOR_EINVAL;
  const thor::HostGrid& gf = fine->grid->h;
  const thor::HostGrid& gc = coarse->grid->h;
  if (nfine != (size_t)gf.ncol || gf.nv != gc.nv) return THOR_EINVAL;
  return fine->precision == THOR_FP64 ? coarse_t<double>(fine, coarse, fine_to_coarse)
                                      : coarse_t<float>(fine, coarse, fine_to_coarse);
}

}  // extern "C"
