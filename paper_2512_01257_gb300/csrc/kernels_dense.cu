// Dense FP64 kernels of the RA-FEAST outer loop (sm_103a).
//
// * Philox-4x64-10 words and Box-Muller normals for Omega (Algorithm 2,
//   "Draw Omega"; Salmon et al., SC'11).
// * Layout moves between the caller's column-major blocks and the internal
//   row-major, row-permuted blocks.
// * Tall-skinny Gram G = X^T Y (Cholesky-QR Gram B_Q = Q~^T Q~ and the
//   Rayleigh-Ritz matrix A_Q = Q^T (A Q), Algorithm 1), split over rows with
//   per-CTA partials and a deterministic second-stage sum.
// * One-CTA Cholesky of the m x m Gram matrix with the shift of shifted
//   Cholesky-QR when it is not numerically positive definite (Fukaya,
//   Kannan, Nakatsukasa, Yamamoto, Yanagisawa, SIAM J. Sci. Comput. 2020),
//   plus the inverse of the triangular factor, so Q = Q~ R^{-1} is a GEMM.
// * Tall GEMM Y = X M (Q R^{-1}, Q V, (A Q) V).
// * One-CTA cyclic Jacobi eigensolver for the reduced symmetric problem
//   (Rayleigh-Ritz, Algorithm 1): round-robin ordering of m/2 disjoint
//   rotations per round, rotation angles from the symmetric 2x2 Schur form.
// * Column norms of A Q - Q diag(theta) (residuals) and column dots.
#include <cfloat>
#include <cmath>

#include "common.cuh"
#include "internal.h"

namespace rafeast {

// ---------------------------------------------------------------------------
// Philox-4x64-10
// ---------------------------------------------------------------------------
__device__ __forceinline__ void philox4x64_10(uint64_t c[4], uint64_t k0, uint64_t k1) {
  const uint64_t M0 = 0xD2E7470EE14C6C93ull, M1 = 0xCA5A826395121157ull;
  const uint64_t W0 = 0x9E3779B97F4A7C15ull, W1 = 0xBB67AE8584CAA73Bull;
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    if (r > 0) {
      k0 += W0;
      k1 += W1;
    }
    const uint64_t hi0 = __umul64hi(M0, c[0]), lo0 = M0 * c[0];
    const uint64_t hi1 = __umul64hi(M1, c[2]), lo1 = M1 * c[2];
    const uint64_t n0 = hi1 ^ c[1] ^ k0, n2 = hi0 ^ c[3] ^ k1;
    c[0] = n0;
    c[1] = lo1;
    c[2] = n2;
    c[3] = lo0;
  }
}

__global__ void k_philox(uint64_t seed, uint64_t first, int64_t nblocks, uint64_t* out) {
  for (int64_t b = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; b < nblocks;
       b += (int64_t)gridDim.x * blockDim.x) {
    uint64_t c[4] = {first + (uint64_t)b, 0, 0, 0};
    philox4x64_10(c, seed, 0);
    out[4 * b + 0] = c[0];
    out[4 * b + 1] = c[1];
    out[4 * b + 2] = c[2];
    out[4 * b + 3] = c[3];
  }
}

__device__ __forceinline__ double u01(uint64_t x) {
  return ((double)(x >> 11) + 1.0) * 0x1.0p-53;
}

// Omega column-major n x k; linear index e = c*n + i; block e/4
__global__ void k_omega(uint64_t seed, int64_t total, double* out) {
  const int64_t nblk = (total + 3) / 4;
  for (int64_t b = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; b < nblk;
       b += (int64_t)gridDim.x * blockDim.x) {
    uint64_t c[4] = {(uint64_t)b, 0, 0, 0};
    philox4x64_10(c, seed, 0);
    double g[4];
    {
      const double rad = sqrt(-2.0 * log(u01(c[0])));
      double s, co;
      sincospi(2.0 * u01(c[1]), &s, &co);
      g[0] = rad * co;
      g[1] = rad * s;
    }
    {
      const double rad = sqrt(-2.0 * log(u01(c[2])));
      double s, co;
      sincospi(2.0 * u01(c[3]), &s, &co);
      g[2] = rad * co;
      g[3] = rad * s;
    }
#pragma unroll
    for (int t = 0; t < 4; ++t)
      if (4 * b + t < total) out[4 * b + t] = g[t];
  }
}

void launch_philox(uint64_t seed, uint64_t first, int64_t nblocks, uint64_t* out,
                   cudaStream_t s) {
  if (nblocks <= 0) return;
  int64_t blocks = (nblocks + 255) / 256;
  if (blocks > 4096) blocks = 4096;
  k_philox<<<(int)blocks, 256, 0, s>>>(seed, first, nblocks, out);
  RF_LAUNCH();
}

void launch_omega(uint64_t seed, int64_t n, int k, double* out, cudaStream_t s) {
  const int64_t total = n * (int64_t)k;
  int64_t blocks = ((total + 3) / 4 + 255) / 256;
  if (blocks > 8192) blocks = 8192;
  if (blocks < 1) blocks = 1;
  k_omega<<<(int)blocks, 256, 0, s>>>(seed, total, out);
  RF_LAUNCH();
}

// ---------------------------------------------------------------------------
// layout moves
// ---------------------------------------------------------------------------
// A CTA moves MV_R rows, consecutive in the caller's order, by MV_C columns
// through shared memory: the column-major side is read or written 32 rows (256 bytes) of a
// column at a time, the row-major side 512 bytes of a row at a time, wherever the
// reordering put it. (One thread per element with the reordered index on the
// column-major side touched a 32-byte sector per 8-byte value: 155 us in and
// 344 us out for 200,000 x 80 against 128 MB each way.)
constexpr int MV_R = 32, MV_C = 64;
__global__ void __launch_bounds__(256) k_to_internal(int64_t n, int m,
                                                     const double* __restrict__ src,
                                                     double* __restrict__ dst, int ld,
                                                     const int32_t* __restrict__ iperm) {
  __shared__ double mv[MV_R][MV_C + 1];
  const int64_t o0 = (int64_t)blockIdx.x * MV_R;
  const int rows = (int)min((int64_t)MV_R, n - o0);
  const int c0 = blockIdx.y * MV_C, nc = min(MV_C, ld - c0);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int u = 0; u < MV_C / 8; ++u) {
    const int c = warp + 8 * u;
    if (c < nc) mv[lane][c] = (c0 + c < m && lane < rows) ? src[(int64_t)(c0 + c) * n + o0 + lane] : 0.0;
  }
  __syncthreads();
  for (int r = warp; r < rows; r += 8) {
    double* out = dst + (iperm ? (int64_t)iperm[o0 + r] : o0 + r) * ld + c0;
    for (int c = lane; c < nc; c += 32) out[c] = mv[r][c];
  }
}

__global__ void __launch_bounds__(256) k_from_internal(int64_t n, int m,
                                                       const double* __restrict__ src, int ld,
                                                       double* __restrict__ dst,
                                                       const int32_t* __restrict__ iperm,
                                                       const int32_t* __restrict__ cols) {
  __shared__ double mv[MV_R][MV_C + 1];
  const int64_t o0 = (int64_t)blockIdx.x * MV_R;
  const int rows = (int)min((int64_t)MV_R, n - o0);
  const int c0 = blockIdx.y * MV_C, nc = min(MV_C, m - c0);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int u = 0; u < MV_R / 8; ++u) {
    const int r = warp + 8 * u;
    if (r >= rows) break;
    const double* in = src + (iperm ? (int64_t)iperm[o0 + r] : o0 + r) * ld;
    for (int c = lane; c < nc; c += 32) mv[r][c] = in[cols ? cols[c0 + c] : c0 + c];
  }
  __syncthreads();
  if (lane < rows)
    for (int c = warp; c < nc; c += 8) dst[(int64_t)(c0 + c) * n + o0 + lane] = mv[lane][c];
}

// the same one element per thread, for blocks that both levels of cache hold
// anyway (at most MV_SMALL elements): no shared-memory phase to wait for. 24
// columns of 2,000 rows: a product with both moves takes 30 us this way, 33 us
// through shared memory; from about 8 MB on the sectors wasted cost more. And for
// blocks of at most MV_NARROW columns at any size, where a CTA's 64 columns would
// be mostly empty and a row is at most four sectors anyway: float product of
// 1,000,000 rows with both moves, one column 153 us against 261, 8 columns 242
// against 322, 14 columns 321 against 379; 200,000 rows 14 columns 119 against
// 122, 16 columns 124 against 121, 24 columns 165 against 150.
constexpr int64_t MV_SMALL = 1 << 19;
constexpr int MV_NARROW = 14;
__global__ void k_to_internal_small(int64_t n, int m, const double* __restrict__ src,
                                    double* __restrict__ dst, int ld,
                                    const int32_t* __restrict__ iperm) {
  const int64_t total = n * (int64_t)ld;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t o = e / ld;
    const int c = (int)(e - o * ld);
    dst[(iperm ? (int64_t)iperm[o] : o) * ld + c] = c < m ? src[(int64_t)c * n + o] : 0.0;
  }
}
__global__ void k_from_internal_small(int64_t n, int m, const double* __restrict__ src, int ld,
                                      double* __restrict__ dst, const int32_t* __restrict__ iperm,
                                      const int32_t* __restrict__ cols) {
  const int64_t total = n * (int64_t)m;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t o = e / m;
    const int c = (int)(e - o * m);
    dst[(int64_t)c * n + o] = src[(iperm ? (int64_t)iperm[o] : o) * ld + (cols ? cols[c] : c)];
  }
}

static int blocks_for(int64_t total, int per = 256, int cap = 16384) {
  int64_t b = (total + per - 1) / per;
  if (b > cap) b = cap;
  if (b < 1) b = 1;
  return (int)b;
}

void launch_to_internal(int64_t n, int m, const double* src, double* dst, int ld,
                        const int32_t* iperm, cudaStream_t s) {
  if (n <= 0 || ld <= 0) return;
  if (n * (int64_t)ld <= MV_SMALL || ld <= MV_NARROW) {
    k_to_internal_small<<<blocks_for(n * (int64_t)ld), 256, 0, s>>>(n, m, src, dst, ld, iperm);
  } else {
    const dim3 grid((unsigned)((n + MV_R - 1) / MV_R), (ld + MV_C - 1) / MV_C);
    k_to_internal<<<grid, 256, 0, s>>>(n, m, src, dst, ld, iperm);
  }
  RF_LAUNCH();
}

void launch_from_internal(int64_t n, int m, const double* src, int ld, double* dst,
                          const int32_t* iperm, const int32_t* cols, cudaStream_t s) {
  if (n <= 0 || m <= 0) return;
  if (n * (int64_t)m <= MV_SMALL || m <= MV_NARROW) {
    k_from_internal_small<<<blocks_for(n * (int64_t)m), 256, 0, s>>>(n, m, src, ld, dst, iperm,
                                                                     cols);
  } else {
    const dim3 grid((unsigned)((n + MV_R - 1) / MV_R), (m + MV_C - 1) / MV_C);
    k_from_internal<<<grid, 256, 0, s>>>(n, m, src, ld, dst, iperm, cols);
  }
  RF_LAUNCH();
}

__global__ void k_cast_f32(const double* __restrict__ src, float* __restrict__ dst, int64_t count) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < count;
       e += (int64_t)gridDim.x * blockDim.x)
    dst[e] = (float)src[e];
}
void launch_cast_to_f32(const double* src, float* dst, int64_t count, cudaStream_t s) {
  if (count <= 0) return;
  k_cast_f32<<<blocks_for(count), 256, 0, s>>>(src, dst, count);
  RF_LAUNCH();
}

__global__ void k_widen(const float* __restrict__ src, double* __restrict__ dst, int64_t count) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < count;
       e += (int64_t)gridDim.x * blockDim.x)
    dst[e] = (double)src[e];
}
void launch_widen(const float* src, double* dst, int64_t count, cudaStream_t s) {
  if (count <= 0) return;
  k_widen<<<blocks_for(count), 256, 0, s>>>(src, dst, count);
  RF_LAUNCH();
}

void launch_zero(void* p, size_t bytes, cudaStream_t s) {
  if (bytes) RF_CUDA(cudaMemsetAsync(p, 0, bytes, s));
}

// ---------------------------------------------------------------------------
// tall-skinny Gram: partial[cta] = X[rows]^T Y[rows], then a column sum
// ---------------------------------------------------------------------------
constexpr int GRAM_RB = 16;

// SYM: the result is symmetric, so the 16-strided tile blocks below the
// diagonal (u > v) are skipped; k_gram_sum mirrors them.
template <int U, bool SYM>
__global__ void __launch_bounds__(256) k_gram_partial(const double* __restrict__ X,
                                                      const double* __restrict__ Y, int64_t n,
                                                      int m, int ld, double* __restrict__ part) {
  extern __shared__ double gsm[];
  double* Xs = gsm;                 // [GRAM_RB][ld]
  double* Ys = gsm + GRAM_RB * ld;  // [GRAM_RB][ld]
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  double acc[U][U];
#pragma unroll
  for (int u = 0; u < U; ++u)
#pragma unroll
    for (int v = 0; v < U; ++v) acc[u][v] = 0.0;
  const int64_t chunk = (n + gridDim.x - 1) / gridDim.x;
  const int64_t r0 = blockIdx.x * chunk;
  const int64_t r1 = min(n, r0 + chunk);
  for (int64_t rb = r0; rb < r1; rb += GRAM_RB) {
    const int rows = (int)min((int64_t)GRAM_RB, r1 - rb);
    __syncthreads();
    for (int t = threadIdx.x; t < GRAM_RB * ld; t += blockDim.x) {
      const int rr = t / ld;
      Xs[t] = rr < rows ? X[(rb + rr) * ld + (t - rr * ld)] : 0.0;
      Ys[t] = rr < rows ? Y[(rb + rr) * ld + (t - rr * ld)] : 0.0;
    }
    __syncthreads();
    for (int rr = 0; rr < rows; ++rr) {
      double xa[U], yb[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int a = tx + 16 * u;
        xa[u] = a < m ? Xs[rr * ld + a] : 0.0;
        const int b = ty + 16 * u;
        yb[u] = b < m ? Ys[rr * ld + b] : 0.0;
      }
#pragma unroll
      for (int u = 0; u < U; ++u)
#pragma unroll
        for (int v = 0; v < U; ++v)
          if (!SYM || u <= v) acc[u][v] = fma(xa[u], yb[v], acc[u][v]);
    }
  }
  double* out = part + (int64_t)blockIdx.x * m * m;
#pragma unroll
  for (int u = 0; u < U; ++u)
#pragma unroll
    for (int v = 0; v < U; ++v) {
      const int a = tx + 16 * u, b = ty + 16 * v;
      if (a < m && b < m && (!SYM || u <= v)) out[a * m + b] = acc[u][v];
    }
}

// X^T X of a preconditioning pass, formed and summed in float within a CTA (the
// CTA partials are added in double): upper tile blocks only. A CTA's rows are one
// run of memory; the next GRAMF_RB rows' 16-byte loads travel in registers during
// this stage's products. A value is rounded to float once, on its way to shared
// memory: conversions issue at the FP64 pipe's rate, and one per use in the
// product loop cost most of the former kernel: a kNN solve of 200,000 x 80 with 14
// such passes took 10 ms more, twelve block-model graphs about 50 ms more.
constexpr int GRAMF_RB = 32;
template <int U>
__global__ void __launch_bounds__(256) k_gram_f32(const double* __restrict__ X, int64_t n, int m,
                                                  int ld, double* __restrict__ part) {
  extern __shared__ float gsf[];  // [GRAMF_RB][ld]
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  float acc[U][U];
#pragma unroll
  for (int u = 0; u < U; ++u)
#pragma unroll
    for (int v = 0; v < U; ++v) acc[u][v] = 0.0f;
  const int64_t chunk = (n + gridDim.x - 1) / gridDim.x;
  const int64_t r0 = blockIdx.x * chunk, r1 = min(n, r0 + chunk);
  constexpr int NV = GRAMF_RB * 16 * U / 2 / 256;  // (ld <= 16 U; at least 1)
  const int pairs = GRAMF_RB * ld / 2;
  double2 nx[NV];
  auto fetch = [&](int64_t rb) {
    const int have = (int)min((int64_t)GRAMF_RB, r1 - rb) * ld / 2;
    const double2* src = reinterpret_cast<const double2*>(X + rb * ld);
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      const int t = threadIdx.x + 256 * v;
      nx[v] = t < have ? src[t] : make_double2(0.0, 0.0);
    }
  };
  if (r0 < r1) fetch(r0);
  for (int64_t rb = r0; rb < r1; rb += GRAMF_RB) {
    __syncthreads();
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      const int t = threadIdx.x + 256 * v;
      if (t < pairs) reinterpret_cast<float2*>(gsf)[t] = make_float2((float)nx[v].x, (float)nx[v].y);
    }
    __syncthreads();
    if (rb + GRAMF_RB < r1) fetch(rb + GRAMF_RB);
    const int rows = (int)min((int64_t)GRAMF_RB, r1 - rb);
#pragma unroll 2
    for (int rr = 0; rr < rows; ++rr) {
      float xa[U], yb[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int a = tx + 16 * u, b = ty + 16 * u;
        xa[u] = a < m ? gsf[rr * ld + a] : 0.0f;
        yb[u] = b < m ? gsf[rr * ld + b] : 0.0f;
      }
#pragma unroll
      for (int u = 0; u < U; ++u)
#pragma unroll
        for (int v = u; v < U; ++v) acc[u][v] = fmaf(xa[u], yb[v], acc[u][v]);
    }
  }
  double* out = part + (int64_t)blockIdx.x * m * m;
#pragma unroll
  for (int u = 0; u < U; ++u)
#pragma unroll
    for (int v = u; v < U; ++v) {
      const int a = tx + 16 * u, b = ty + 16 * v;
      if (a < m && b < m) out[a * m + b] = (double)acc[u][v];
    }
}

// sym: entries (a, b) with a / 16 > b / 16 were not computed; take (b, a).
// The partials are added in increasing order with Neumaier's compensated
// summation (A. Neumaier, ZAMM 54, 1974): the rounding error of every
// addition is carried along, so the sum of the CTAs' partials adds about
// two units of rounding instead of one per partial.
// Eight lanes share an entry: lane l adds the partials l, l + 8, ..., then the
// lanes' (sum, error) pairs are added by a fixed tree. (One thread per entry
// ran a chain of 152 or 304 dependent FP64 additions: 63 to 117 us for m = 52
// to 100.)
__global__ void __launch_bounds__(128) k_gram_sum(const double* __restrict__ part, int nparts,
                                                  int m, int sym, double* G) {
  const int mm = m * m;
  const int e = blockIdx.x * 16 + (threadIdx.x >> 3), l = threadIdx.x & 7;
  const bool on = e < mm;
  const int a = on ? e / m : 0, b = on ? e - a * m : 0;
  const int src = (sym && (a >> 4) > (b >> 4)) ? b * m + a : (on ? e : 0);
  double s = 0.0, c = 0.0;
  auto add = [&](double v) {
    const double t = s + v;
    c += fabs(s) >= fabs(v) ? (s - t) + v : (v - t) + s;
    s = t;
  };
  for (int p0 = l; p0 < nparts; p0 += 64) {
    double v[8];  // (past the end: + 0, which changes nothing)
#pragma unroll
    for (int u = 0; u < 8; ++u)
      v[u] = p0 + 8 * u < nparts ? part[(int64_t)(p0 + 8 * u) * mm + src] : 0.0;
#pragma unroll
    for (int u = 0; u < 8; ++u) add(v[u]);
  }
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) {
    const double so = __shfl_xor_sync(0xffffffffu, s, o), co = __shfl_xor_sync(0xffffffffu, c, o);
    // (the lower lane's pair first, so that all lanes of an entry agree)
    const double x = (l & o) ? so : s, y = (l & o) ? s : so;
    c = (l & o) ? co + c : c + co;
    s = x;
    add(y);
  }
  if (on && l == 0) G[e] = s + c;
}

int gram_parts(int num_sms) { return 2 * num_sms; }

void gram_sum(const double* part, int parts, int m, bool sym, double* G, cudaStream_t s) {
  k_gram_sum<<<(m * m + 15) / 16, 128, 0, s>>>(part, parts, m, sym ? 1 : 0, G);
  RF_LAUNCH();
}

template <bool SYM>
static void gram_partials(const double* X, const double* Y, int64_t n, int m, int ld,
                          double* partial, int parts, size_t smem, cudaStream_t s) {
  switch ((m + 15) / 16) {
#define RF_GRAM(UU)                                                                      \
  case UU:                                                                               \
    ensure_dyn_smem(reinterpret_cast<const void*>(k_gram_partial<UU, SYM>), smem);      \
    k_gram_partial<UU, SYM><<<parts, 256, smem, s>>>(X, Y, n, m, ld, partial);           \
    break;
    RF_GRAM(1) RF_GRAM(2) RF_GRAM(3) RF_GRAM(4) RF_GRAM(5) RF_GRAM(6) RF_GRAM(7) RF_GRAM(8)
#undef RF_GRAM
    default: throw Err{RAFEAST_ERR_INVALID_ARG};
  }
}

static void gram_f32(const double* X, int64_t n, int m, int ld, double* partial, int parts,
                     cudaStream_t s) {
  RF_CHECK(ld % 2 == 0 && ld <= (m + 15) / 16 * 16, RAFEAST_ERR_INVALID_ARG);
  const size_t smem = GRAMF_RB * (size_t)ld * sizeof(float);
  switch ((m + 15) / 16) {
#define RF_GRAMF(UU) \
  case UU: k_gram_f32<UU><<<parts, 256, smem, s>>>(X, n, m, ld, partial); break;
    RF_GRAMF(1) RF_GRAMF(2) RF_GRAMF(3) RF_GRAMF(4) RF_GRAMF(5) RF_GRAMF(6) RF_GRAMF(7) RF_GRAMF(8)
#undef RF_GRAMF
    default: throw Err{RAFEAST_ERR_INVALID_ARG};
  }
}

void gram(const double* X, const double* Y, int64_t n, int m, int ld, double* G,
          double* partial, int num_sms, cudaStream_t s, bool sym, bool f32) {
  const int parts = gram_parts(num_sms);
  const size_t smem = 2 * GRAM_RB * (size_t)ld * sizeof(double);
  if (f32) {
    // only the symmetric X^T X of a preconditioning pass is formed in float
    if (!sym) throw Err{RAFEAST_ERR_INVALID_ARG};
    gram_f32(X, n, m, ld, partial, parts, s);
  } else if (sym) {
    gram_partials<true>(X, Y, n, m, ld, partial, parts, smem, s);
  } else {
    gram_partials<false>(X, Y, n, m, ld, partial, parts, smem, s);
  }
  RF_LAUNCH();
  gram_sum(partial, parts, m, sym, G, s);
}

// ---------------------------------------------------------------------------
// tall GEMM: Y[r][b] = sum_a X[r][a] M[a][b]   (M row-major m x mo)
// ---------------------------------------------------------------------------
// A row of Y is computed by L = ceil(mo / V) threads, V columns each
// (b = lane + L v), so that few lanes idle when mo is not a multiple of 32
// (mo = 80: 27 lanes, 81 slots); a CTA of 256 threads takes 256 / L rows
// (at most GEMM_MAX_ROWS) per tile. Rows of a tile may straddle warps.
constexpr int GEMM_MAX_ROWS = 32;

// UPPER: M is upper triangular (M[a][b] = 0 for a > b): column block v
// (b < L v + L) needs rows a < L v + L only, a bound shared by the row's lanes
template <int V, bool UPPER>
__global__ void __launch_bounds__(256) k_tall_gemm(const double* __restrict__ X, int64_t n, int m,
                                                   int ldx, const double* __restrict__ M, int mo,
                                                   double* __restrict__ Y, int ldy) {
  extern __shared__ double tsm[];
  const int L = (mo + V - 1) / V;
  const int rpt = min(GEMM_MAX_ROWS, (int)blockDim.x / L);  // rows per tile
  double* Ms = tsm;              // m * mo
  double* Xs = tsm + m * mo;     // rpt * m
  for (int t = threadIdx.x; t < m * mo; t += blockDim.x) Ms[t] = M[t];
  const int tr = threadIdx.x / L, tc = threadIdx.x - (threadIdx.x / L) * L;
  for (int64_t rb = blockIdx.x * (int64_t)rpt; rb < n; rb += (int64_t)gridDim.x * rpt) {
    __syncthreads();
    const int rows = (int)min((int64_t)rpt, n - rb);
    for (int t = threadIdx.x; t < rpt * m; t += blockDim.x) {
      const int rr = t / m;
      Xs[t] = rr < rows ? X[(rb + rr) * ldx + (t - rr * m)] : 0.0;
    }
    __syncthreads();
    if (tr < rows) {
      double acc[V];
#pragma unroll
      for (int v = 0; v < V; ++v) acc[v] = 0.0;
      for (int a = 0; a < m; ++a) {
        const double x = Xs[tr * m + a];
#pragma unroll
        for (int v = 0; v < V; ++v) {
          const int b = tc + L * v;
          if (UPPER && a >= L * v + L) continue;
          if (b < mo) acc[v] = fma(x, Ms[a * mo + b], acc[v]);
        }
      }
#pragma unroll
      for (int v = 0; v < V; ++v) {
        const int b = tc + L * v;
        if (b < mo) Y[(rb + tr) * ldy + b] = acc[v];
      }
    }
  }
}

void tall_gemm(const double* X, int64_t n, int m, int ldx, const double* M, int mo, double* Y,
               int ldy, cudaStream_t s, bool upper) {
  const int V = (mo + 31) / 32;
  const int L = (mo + V - 1) / V;
  const int rpt = std::min(GEMM_MAX_ROWS, 256 / L);
  const size_t smem = ((size_t)m * mo + (size_t)rpt * m) * sizeof(double);
  int dev = 0, sms = 0;
  RF_CUDA(cudaGetDevice(&dev));
  RF_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  const int64_t tiles = (n + rpt - 1) / rpt;
  int blocks = (int)std::min<int64_t>(tiles, (int64_t)sms * 2);
  if (blocks < 1) blocks = 1;
  switch (V) {
#define RF_TG(VV)                                                                     \
  case VV:                                                                            \
    if (upper) {                                                                      \
      ensure_dyn_smem(reinterpret_cast<const void*>(k_tall_gemm<VV, true>), smem);   \
      k_tall_gemm<VV, true><<<blocks, 256, smem, s>>>(X, n, m, ldx, M, mo, Y, ldy);   \
    } else {                                                                          \
      ensure_dyn_smem(reinterpret_cast<const void*>(k_tall_gemm<VV, false>), smem);  \
      k_tall_gemm<VV, false><<<blocks, 256, smem, s>>>(X, n, m, ldx, M, mo, Y, ldy);  \
    }                                                                                 \
    break;
    RF_TG(1) RF_TG(2) RF_TG(3) RF_TG(4)
#undef RF_TG
    default: throw Err{RAFEAST_ERR_INVALID_ARG};
  }
  RF_LAUNCH();
}

// ---------------------------------------------------------------------------
// Cholesky (+shift) by one CTA, then the triangular inverse by one warp per
// column. G: m x m (row-major, symmetric). Outputs R (upper, G = R^T R,
// row-major) and Rinv (upper, row-major); status: 0 ok, 1 shifted, 2 failed.
//
// One SM issues 2 FP64 lane operations a clock, so the m^3 / 6 products of the
// factorisation alone take 22 us at m = 80; the inverse, as many again, is
// spread over the chip, where a column costs a latency chain of m steps. (Both
// in one CTA, the inverse one column per thread: 441 us in the launch list of the
// kNN solve, 80 and 100 columns; now 170 and 29 us.)
// ---------------------------------------------------------------------------
// a / b from the rounded reciprocal ib: one step on the residual rounds the product
// as the quotient (P. Markstein, IBM J. Res. Develop. 34, 1990); a ib alone has a
// second rounding. Orthonormalising 2,000 x 80 takes 670 us this way (632 with one
// rounding more, 789 with a division per entry), 200,000 x 80 3429 (3391, 3561).
__device__ __forceinline__ double over(double a, double b, double ib) {
  const double q = a * ib;
  return fma(fma(-q, b, a), ib, q);
}

// S: column-major lower triangle, S[k * m + i] = L_ik (i >= k)
__device__ bool chol_inplace(double* S, int m) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  __shared__ int s_bad;
  if (threadIdx.x == 0) s_bad = 0;
  __syncthreads();
  for (int k = 0; k < m; ++k) {
    double* Sk = S + k * m;
    if (warp == 0) {  // the pivot, computed by every lane, and its column
      const double d = Sk[k];
      const bool bad = !(d > 0.0) || !isfinite(d);
      const double r = sqrt(d), ir = 1.0 / r;
      __syncwarp();
      if (lane == 0) {
        if (bad) s_bad = 1;
        else Sk[k] = r;
      }
      if (!bad)
        for (int i = k + 1 + lane; i < m; i += 32) Sk[i] = over(Sk[i], r, ir);
    }
    __syncthreads();
    if (s_bad) return false;
    // trailing update, a warp per column
    for (int j = k + 1 + warp; j < m; j += nw) {
      const double ljk = Sk[j];
      for (int i = j + lane; i < m; i += 32) S[j * m + i] = fma(-Sk[i], ljk, S[j * m + i]);
    }
    __syncthreads();
  }
  return true;
}

__global__ void __launch_bounds__(512) k_chol(const double* __restrict__ G, int m,
                                              double shift_scale, double* __restrict__ R,
                                              int* status, int check_id) {
  extern __shared__ double S[];  // m*m
  __shared__ double s_shift;
  __shared__ int s_far;
  if (threadIdx.x == 0) s_far = 0;
  __syncthreads();
  for (int t = threadIdx.x; t < m * m; t += blockDim.x) {
    S[t] = G[t];
    // check_id: G is the Gram of a block that should be close to orthonormal;
    // flag (status bit 4) when an entry is off the identity by more than 1/4
    if (check_id && fabs(G[t] - ((t / m == t % m) ? 1.0 : 0.0)) > 0.25) s_far = 1;
  }
  __syncthreads();
  int st = 0;
  bool ok = chol_inplace(S, m);
  if (!ok) {
    // shifted Cholesky-QR: s = 11 (n m + m (m + 1)) u ||X||_2^2, ||X||_2^2 <= trace(G)
    __syncthreads();
    if (threadIdx.x == 0) {
      double tr = 0.0;
      for (int i = 0; i < m; ++i) tr += fabs(G[i * m + i]);
      s_shift = shift_scale * tr;
    }
    __syncthreads();
    for (int t = threadIdx.x; t < m * m; t += blockDim.x) {
      const int i = t / m, j = t % m;
      S[t] = G[t] + (i == j ? s_shift : 0.0);
    }
    __syncthreads();
    ok = chol_inplace(S, m);
    st = ok ? 1 : 2;
  }
  if (!ok) {
    if (threadIdx.x == 0) status[0] = 2;
    return;
  }
  // R = L^T: row k of R is column k of L
  for (int t = threadIdx.x; t < m * m; t += blockDim.x) R[t] = t % m >= t / m ? S[t] : 0.0;
  if (threadIdx.x == 0) status[0] = st | (s_far ? 4 : 0);
}

// column j of L^-1 (row j of Rinv) by forward substitution, one warp: lane l
// holds the entries l, l + 32, ... of the right-hand side, column i of L
// (row i of R) leaves it once x_i is known
__global__ void __launch_bounds__(32) k_trinv(const double* __restrict__ R, int m,
                                              double* __restrict__ Rinv, const int* status) {
  if (status[0] == 2) return;
  const int j = blockIdx.x, lane = threadIdx.x;
  double b[4], dg[4], id[4];
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int i = lane + 32 * u;
    b[u] = i == j ? 1.0 : 0.0;
    dg[u] = i < m ? R[i * m + i] : 1.0;
    id[u] = 1.0 / dg[u];
  }
  double l[4], ln[4];
#pragma unroll
  for (int u = 0; u < 4; ++u) l[u] = lane + 32 * u < m ? R[j * m + lane + 32 * u] : 0.0;
  for (int i = j; i < m; ++i) {
#pragma unroll
    for (int u = 0; u < 4; ++u)
      ln[u] = (i + 1 < m && lane + 32 * u < m) ? R[(i + 1) * m + lane + 32 * u] : 0.0;
    const int u0 = i >> 5;
    const double xb = u0 == 0   ? over(b[0], dg[0], id[0])
                      : u0 == 1 ? over(b[1], dg[1], id[1])
                      : u0 == 2 ? over(b[2], dg[2], id[2])
                                : over(b[3], dg[3], id[3]);
    const double x = __shfl_sync(0xffffffffu, xb, i & 31);
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int r = lane + 32 * u;
      if (r == i) b[u] = x;
      else if (r > i) b[u] = fma(-l[u], x, b[u]);
      l[u] = ln[u];
    }
  }
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int i = lane + 32 * u;
    if (i < m) Rinv[j * m + i] = i >= j ? b[u] : 0.0;
  }
}

void chol_inv(double* G, int m, int64_t nrows, double* Rfac, double* Rinv, int* status,
              cudaStream_t s, bool check_id) {
  RF_CHECK(m >= 1 && m <= 128, RAFEAST_ERR_INVALID_ARG);
  const size_t smem = (size_t)m * m * sizeof(double);
  ensure_dyn_smem(reinterpret_cast<const void*>(k_chol), smem);
  const double u = DBL_EPSILON / 2;
  const double scale = 11.0 * ((double)nrows * m + (double)m * (m + 1)) * u;
  k_chol<<<1, 512, smem, s>>>(G, m, scale, Rfac, status, check_id ? 1 : 0);
  RF_LAUNCH();
  k_trinv<<<m, 32, 0, s>>>(Rfac, m, Rinv, status);
  RF_LAUNCH();
}

// ---------------------------------------------------------------------------
// one-CTA cyclic Jacobi (round-robin parallel order), in precision T
// ---------------------------------------------------------------------------
constexpr size_t JACOBI_SMEM_MAX = 216 * 1024;  // A and V in shared memory up to this size

// A (m x m, ld m, symmetric part taken) -> eigenvalues ascending in w, the
// matching eigenvectors as the columns of Vout (m x m, ld m). A pair (p, q)
// is rotated while |a_pq| > rot_tol sqrt(|a_pp a_qq|); the sweeps end when
// the off-diagonal mass is below off_tol of the total or a sweep rotated
// nothing. An entry below abs_tol times the root mean square eigenvalue is left
// alone where the pair's eigenvalues are over JACOBI_CLOSE times as far apart: it
// moves them by less than |a_pq| / JACOBI_CLOSE. In a closer pair it moves them by
// up to |a_pq| and counts however small it is (three rows with a pair at 2^-30
// joined by 2^-51: the pair's error with the absolute rule alone was 2^-51).
// Vg: global fallback for the eigenvector accumulator (me * me), which is kept
// transposed (an entry's column-wise neighbours in V, 16 lanes of a warp in one
// shared-memory bank, made a float round of m = 80 three times as long).
constexpr double JACOBI_CLOSE = 64.0;
template <typename T>
__global__ void __launch_bounds__(1024) k_jacobi(const double* __restrict__ Ain, int m, double* __restrict__ w,
                         double* __restrict__ Vout, T* __restrict__ Vg, int max_sweeps,
                         double rot_tol, double off_tol, double abs_tol) {
  extern __shared__ unsigned char jsm[];
  T* A = reinterpret_cast<T*>(jsm);  // me * me (+ me * me for V when it fits)
  const int me = m + (m & 1);
  // the eigenvector accumulator in shared memory when both fit, else in the
  // global work buffer
  T* Vw = (2 * (size_t)me * me * sizeof(T) <= JACOBI_SMEM_MAX) ? A + me * me : Vg;
  __shared__ T cs[64 * 2];  // c, s per pair (me/2 <= 64)
  __shared__ int pq[64 * 2];
  __shared__ double s_off, s_tot;
  __shared__ double s_woff[32], s_wtot[32];  // per-warp sums, added in warp order
  __shared__ int s_order[128];
  __shared__ int s_rot;
  const T tiny = sizeof(T) == 4 ? (T)1e-37 : (T)1e-300;
  for (int t = threadIdx.x; t < me * me; t += blockDim.x) {
    const int i = t / me, j = t % me;
    A[t] = (i < m && j < m) ? (T)(0.5 * (Ain[i * m + j] + Ain[j * m + i])) : (T)0;
    Vw[t] = (i == j) ? (T)1 : (T)0;
  }
  __syncthreads();
  const int np = me / 2;
  // this thread's 2 x 2 blocks (j, k) of A and entries (k, row) of V^T are the
  // same in every round
  constexpr int TA = 4, TV = 8;  // np * np <= 4 * 1024, np * me <= 8 * 1024
  int tj[TA], tk[TA], vk[TV], vr[TV];
#pragma unroll
  for (int u = 0; u < TA; ++u) {
    const int t = threadIdx.x + u * (int)blockDim.x;
    tj[u] = t < np * np ? t / np : -1;
    tk[u] = t - (t / np) * np;
  }
#pragma unroll
  for (int u = 0; u < TV; ++u) {
    const int t = threadIdx.x + u * (int)blockDim.x;
    vk[u] = t < np * me ? t / me : -1;
    vr[u] = t - (t / me) * me;
  }
  for (int sweep = 0; sweep < max_sweeps; ++sweep) {
    // convergence test on the off-diagonal mass
    if (threadIdx.x == 0) {
      s_off = 0.0;
      s_tot = 0.0;
      s_rot = 0;
    }
    __syncthreads();
    double off = 0.0, tot = 0.0;
    for (int t = threadIdx.x; t < me * me; t += blockDim.x) {
      const int i = t / me, j = t % me;
      const double a2 = (double)A[t] * (double)A[t];
      tot += a2;
      if (i != j) off += a2;
    }
    off = warp_sum(off);
    tot = warp_sum(tot);
    if ((threadIdx.x & 31) == 0) {
      s_woff[threadIdx.x >> 5] = off;
      s_wtot[threadIdx.x >> 5] = tot;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      double so = 0.0, st = 0.0;
      for (int wi = 0; wi < (int)(blockDim.x >> 5); ++wi) {
        so += s_woff[wi];
        st += s_wtot[wi];
      }
      s_off = so;
      s_tot = st;
    }
    __syncthreads();
    if (!(s_off > off_tol * s_tot) || s_tot == 0.0) break;
    const T small = (T)(abs_tol * sqrt(s_tot / m));
    // a_pq is worth a rotation (the square root, an FP64 chain, comes last)
    auto counts = [&](T apq, T app, T aqq) {
      const T x = fabs(apq);
      return x > tiny && (x > small || x * (T)JACOBI_CLOSE > fabs(app - aqq)) &&
             x > (T)rot_tol * sqrt(fabs(app * aqq));
    };
    if (abs_tol > 0.0) {  // no sweep for what is left of the refined matrix, as a rule
      int any = 0;
      for (int t = threadIdx.x; t < me * me; t += blockDim.x) {
        const int i = t / me, j = t % me;
        if (i < j) any |= counts(A[t], A[i * me + i], A[j * me + j]) ? 1 : 0;
      }
      if (!__syncthreads_or(any)) break;
    }
    for (int round = 0; round < me - 1; ++round) {
      int rotates = 0;
      for (int k = threadIdx.x; k < np; k += blockDim.x) {
        // circle method: position 0 fixed, others rotate
        auto player = [&](int pos) {
          const int x = pos - 1 + round;  // < 2 (me - 1)
          return pos == 0 ? 0 : (x >= me - 1 ? x - (me - 1) : x) + 1;
        };
        int p = player(k), q = player(me - 1 - k);
        if (p > q) {
          const int t = p;
          p = q;
          q = t;
        }
        const T apq = A[p * me + q];
        T c = (T)1, s = (T)0;
        const T app = A[p * me + p], aqq = A[q * me + q];
        if (counts(apq, app, aqq)) {
          s_rot = 1;
          rotates = 1;
          const T tau = (aqq - app) / ((T)2 * apq);
          const T at = fabs(tau);
          const T root = at > (T)1e15 ? at : sqrt((T)1 + tau * tau);
          const T t = (tau >= (T)0 ? (T)1 : (T)-1) / (at + root);
          c = (T)1 / sqrt((T)1 + t * t);
          s = t * c;
        }
        cs[2 * k] = c;
        cs[2 * k + 1] = s;
        pq[2 * k] = p;
        pq[2 * k + 1] = q;
      }
      if (!__syncthreads_or(rotates)) continue;  // (no pair of this round is rotated)
      // the pairs of a round are disjoint, so every 2 x 2 block (rows of
      // pair j, columns of pair k) is updated on its own from its old
      // values: B <- L_j B R_k with L = [[c, -s], [s, c]], R = L^T; the
      // rotated diagonal blocks lose their off-diagonal entry
#pragma unroll
      for (int u = 0; u < TA; ++u) {
        if (tj[u] < 0) break;
        const int j = tj[u], k = tk[u];
        const T cj = cs[2 * j], sj = cs[2 * j + 1];
        const T ck = cs[2 * k], sk = cs[2 * k + 1];
        if (sj == (T)0 && sk == (T)0) continue;
        const int pj = pq[2 * j], qj = pq[2 * j + 1];
        const int pk = pq[2 * k], qk = pq[2 * k + 1];
        const T a11 = A[pj * me + pk], a12 = A[pj * me + qk];
        const T a21 = A[qj * me + pk], a22 = A[qj * me + qk];
        // rows: L_j B
        const T b11 = cj * a11 - sj * a21, b12 = cj * a12 - sj * a22;
        const T b21 = sj * a11 + cj * a21, b22 = sj * a12 + cj * a22;
        // columns: (L_j B) R_k
        A[pj * me + pk] = ck * b11 - sk * b12;
        A[pj * me + qk] = j == k ? (T)0 : sk * b11 + ck * b12;
        A[qj * me + pk] = j == k ? (T)0 : ck * b21 - sk * b22;
        A[qj * me + qk] = sk * b21 + ck * b22;
      }
      // V R_k, on V^T: a warp's lanes take consecutive entries of the two rows
#pragma unroll
      for (int u = 0; u < TV; ++u) {
        if (vk[u] < 0) break;
        const int k = vk[u], row = vr[u];
        const T c = cs[2 * k], s = cs[2 * k + 1];
        if (s == (T)0) continue;
        const int p = pq[2 * k], q = pq[2 * k + 1];
        const T vp = Vw[p * me + row], vq = Vw[q * me + row];
        Vw[p * me + row] = c * vp - s * vq;
        Vw[q * me + row] = s * vp + c * vq;
      }
      __syncthreads();
    }
    if (s_rot == 0) break;  // nothing was above the threshold in this sweep
    __syncthreads();
  }
  // eigenvalues ascending (m <= 128; equal ones in index order): the rank of
  // each; then w and the columns of V
  __syncthreads();
  for (int i = threadIdx.x; i < m; i += blockDim.x) s_order[i] = i;  // (kept where NaNs leave a gap)
  __syncthreads();
  for (int i = threadIdx.x; i < m; i += blockDim.x) {
    const T v = A[i * me + i];
    int rank = 0;
    for (int j = 0; j < m; ++j) {
      const T x = A[j * me + j];
      rank += (x < v || (x == v && j < i)) ? 1 : 0;
    }
    s_order[rank] = i;
  }
  __syncthreads();
  for (int i = threadIdx.x; i < m; i += blockDim.x) w[i] = (double)A[s_order[i] * me + s_order[i]];
  for (int t = threadIdx.x; t < m * m; t += blockDim.x) {
    const int r = t / m, c = t % m;
    Vout[r * m + c] = (double)Vw[s_order[c] * me + r];
  }
}

// small dense product, all m x m row-major: C = alpha op(A) op(B) + gamma I,
// op = transpose when the flag is set. A CTA of 64 threads forms an 8 x 8
// block of C from panels staged in shared memory: small blocks put the FP64
// work (2 lane operations per SM and clock) on every SM (18 us with one entry
// per thread of 128 and the operands read from global memory, m = 80).
__global__ void __launch_bounds__(64) k_small_gemm(const double* __restrict__ A, int ta,
                                                   const double* __restrict__ B, int tb,
                                                   double* __restrict__ C, int m, double alpha,
                                                   double gamma) {
  __shared__ double sa[8][129], sb[8][129];  // rows of op(A), columns of op(B)
  const int i0 = blockIdx.y * 8, j0 = blockIdx.x * 8;
  for (int t = threadIdx.x; t < 8 * m; t += 64) {
    // (consecutive threads along the operand's contiguous dimension)
    const int ra = ta ? t % 8 : t / m, ka = ta ? t / 8 : t % m;
    const int rb = tb ? t / m : t % 8, kb = tb ? t % m : t / 8;
    sa[ra][ka] = i0 + ra < m ? (ta ? A[ka * m + i0 + ra] : A[(i0 + ra) * m + ka]) : 0.0;
    sb[rb][kb] = j0 + rb < m ? (tb ? B[(j0 + rb) * m + kb] : B[kb * m + j0 + rb]) : 0.0;
  }
  __syncthreads();
  const int i = threadIdx.x >> 3, j = threadIdx.x & 7;
  double acc = 0.0;
#pragma unroll 4
  for (int k = 0; k < m; ++k) acc = fma(sa[i][k], sb[j][k], acc);
  if (i0 + i < m && j0 + j < m)
    C[(i0 + i) * m + j0 + j] = alpha * acc + (i0 + i == j0 + j ? gamma : 0.0);
}

void small_gemm(const double* A, int ta, const double* B, int tb, double* C, int m, double alpha,
                double gamma, cudaStream_t s) {
  RF_CHECK(m >= 1 && m <= 128, RAFEAST_ERR_INVALID_ARG);
  const dim3 grid((m + 7) / 8, (m + 7) / 8);
  k_small_gemm<<<grid, 64, 0, s>>>(A, ta, B, tb, C, m, alpha, gamma);
  RF_LAUNCH();
}

template <typename T>
static void jacobi_launch(const double* A, int m, double* w, double* V, T* Vg, int sweeps,
                          double rot_tol, double off_tol, double abs_tol, cudaStream_t s) {
  const int me = m + (m & 1);
  size_t smem = (size_t)me * me * sizeof(T);
  if (2 * smem <= JACOBI_SMEM_MAX) smem *= 2;  // V beside A
  ensure_dyn_smem(reinterpret_cast<const void*>(k_jacobi<T>), smem);
  k_jacobi<T><<<1, 1024, smem, s>>>(A, m, w, V, Vg, sweeps, rot_tol, off_tol, abs_tol);
  RF_LAUNCH();
}

// U = I + E of a nearly diagonal symmetric B: the first-order rotations
// e_ij = b_ij / (b_jj - b_ii) (Jacobi 1846; the separated case of Ogita and
// Aishima, "Iterative refinement for symmetric eigenvalue decomposition", Japan
// J. Indust. Appl. Math. 35, 2018). A pair with |e_ij| > 0.02 (a cluster) is
// left to the Jacobi sweeps that follow, and so are all pairs of a row whose
// |e_ij| add up to more than 0.1: ||E|| <= 0.1, and three Newton-Schulz steps
// bring U^T U from I + 1e-2 to I + 2e-17. One CTA per row; full[i]: row i is
// over the sum.
__device__ __forceinline__ double first_order(const double* __restrict__ B, int m, int i, int j) {
  if (i == j) return 0.0;
  const double b = 0.5 * (B[i * m + j] + B[j * m + i]);
  const double gap = B[j * m + j] - B[i * m + i];
  return fabs(b) <= 0.02 * fabs(gap) && gap != 0.0 ? b / gap : 0.0;
}
__global__ void __launch_bounds__(128) k_first_order_sums(const double* __restrict__ B, int m,
                                                          int* __restrict__ full) {
  __shared__ double sw[4];
  const int i = blockIdx.x;
  const double e = threadIdx.x < m ? fabs(first_order(B, m, i, threadIdx.x)) : 0.0;
  const double t = warp_sum(e);
  if ((threadIdx.x & 31) == 0) sw[threadIdx.x >> 5] = t;
  __syncthreads();
  if (threadIdx.x == 0) full[i] = !(sw[0] + sw[1] + sw[2] + sw[3] <= 0.1);
}
__global__ void __launch_bounds__(128) k_first_order(const double* __restrict__ B, int m,
                                                     const int* __restrict__ full,
                                                     double* __restrict__ U) {
  const int i = blockIdx.x, j = threadIdx.x;
  if (j >= m) return;
  U[i * m + j] = i == j ? 1.0 : (full[i] || full[j]) ? 0.0 : first_order(B, m, i, j);
}

// the three rounds of jacobi_eigh's step (3) for m <= REFINE_M in one CTA, one thread
// per entry and every matrix in shared memory; the sums are those of k_small_gemm.
// 33 dependent launches of 2 to 3 us are longer than the arithmetic of small
// matrices: a Rayleigh-Ritz call of 2,000 rows with 1, 4, 8 and 16 columns
// took 289, 373, 405 and 473 us with them and takes 201, 266, 309 and 414 us.
constexpr int REFINE_M = 16;
__global__ void __launch_bounds__(REFINE_M * REFINE_M) k_refine_small(double* __restrict__ Bg,
                                                                      double* __restrict__ Wg, int m) {
  using Mat = double[REFINE_M][REFINE_M + 1];
  __shared__ Mat B, W, U, S;
  __shared__ int full[REFINE_M];
  const int i = threadIdx.x / REFINE_M, j = threadIdx.x % REFINE_M;
  const bool on = i < m && j < m;
  B[i][j] = on ? Bg[i * m + j] : 0.0;
  W[i][j] = on ? Wg[i * m + j] : 0.0;
  __syncthreads();
  auto first = [&](int r, int c) {  // first_order on the padded rows
    if (r == c) return 0.0;
    const double b = 0.5 * (B[r][c] + B[c][r]), gap = B[c][c] - B[r][r];
    return fabs(b) <= 0.02 * fabs(gap) && gap != 0.0 ? b / gap : 0.0;
  };
  // C = alpha op(X) Y + gamma I (every thread has its entry before any is stored)
  auto gemm = [&](const Mat& X, bool tx, const Mat& Y, Mat& C, double alpha, double gamma) {
    double acc = 0.0;
    for (int k = 0; k < m; ++k) acc = fma(tx ? X[k][i] : X[i][k], Y[k][j], acc);
    __syncthreads();
    if (on) C[i][j] = alpha * acc + (i == j ? gamma : 0.0);
    __syncthreads();
  };
  for (int it = 0; it < 3; ++it) {
    if (j == 0 && i < m) {
      double t = 0.0;
      for (int c = 0; c < m; ++c) t += fabs(first(i, c));
      full[i] = !(t <= 0.1);
    }
    __syncthreads();
    if (on) U[i][j] = i == j ? 1.0 : (full[i] || full[j]) ? 0.0 : first(i, j);
    __syncthreads();
    for (int ns = 0; ns < 3; ++ns) {
      gemm(U, true, U, S, -0.5, 1.5);
      gemm(U, false, S, U, 1.0, 0.0);
    }
    gemm(B, false, U, S, 1.0, 0.0);
    gemm(U, true, S, B, 1.0, 0.0);
    gemm(W, false, U, W, 1.0, 0.0);
  }
  if (on) {
    Bg[i * m + j] = B[i][j];
    Wg[i * m + j] = W[i][j];
  }
}

// Mixed-precision Jacobi. GB300's FP64 rate is a small fraction of its FP32
// rate, and a one-CTA FP64 Jacobi sweep of an 80 x 80 matrix takes 0.8 ms of
// one SM's FP64 issue. So: (1) float Jacobi to the float rounding floor gives
// V1 with V1^T A V1 diagonal to ~1e-7; (2) two Newton-Schulz steps
// V <- V (3 I - V^T V) / 2 make V1 orthonormal to working precision (its
// float error is ~1e-6, each step squares it); (3) three rounds of first-order
// rotations on B = V1^T A V1, U = I + E made orthonormal by three Newton-Schulz
// steps, square its off-diagonal part for every pair that is not a cluster, by
// products that run on all SMs; (4) FP64 Jacobi sweeps on what is left, none
// when every entry is within a few units of rounding (8 eps of the root mean
// square eigenvalue) and no close pair is coupled; (5) V = V1 U1 U2 U3 V_B. On the
// kNN Rayleigh-Ritz matrix of 80 columns the FP64 part took 2.2 ms as Jacobi sweeps
// alone.
void jacobi_eigh(double* A, int m, double* w, double* V, double* work, cudaStream_t s) {
  if (m > 128) throw Err{RAFEAST_ERR_INVALID_ARG};
  const int me = m + (m & 1);
  const size_t mm = (size_t)me * me;
  double* W1 = work;
  double* W2 = work + mm;
  double* S = work + 2 * mm;
  double* B = work + 3 * mm;
  double* VB = work + 4 * mm;
  double* Vg = work + 5 * mm;  // also the float stage's fallback accumulator
  jacobi_launch<float>(A, m, w, W1, reinterpret_cast<float*>(Vg), 30, 1e-6, 1e-13, 0.0, s);
  for (int it = 0; it < 2; ++it) {
    small_gemm(W1, 1, W1, 0, S, m, -0.5, 1.5, s);  // S = (3 I - V^T V) / 2
    small_gemm(W1, 0, S, 0, W2, m, 1.0, 0.0, s);   // V <- V S
    std::swap(W1, W2);
  }
  small_gemm(A, 0, W1, 0, S, m, 1.0, 0.0, s);  // A V
  small_gemm(W1, 1, S, 0, B, m, 1.0, 0.0, s);  // V^T A V
  if (m <= REFINE_M) {
    k_refine_small<<<1, REFINE_M * REFINE_M, 0, s>>>(B, W1, m);
    RF_LAUNCH();
  }
  for (int it = 0; it < 3 && m > REFINE_M; ++it) {
    k_first_order_sums<<<m, 128, 0, s>>>(B, m, reinterpret_cast<int*>(S));
    RF_LAUNCH();
    k_first_order<<<m, 128, 0, s>>>(B, m, reinterpret_cast<const int*>(S), VB);
    RF_LAUNCH();
    for (int ns = 0; ns < 3; ++ns) {
      small_gemm(VB, 1, VB, 0, S, m, -0.5, 1.5, s);  // (3 I - U^T U) / 2
      small_gemm(VB, 0, S, 0, Vg, m, 1.0, 0.0, s);   // U
      std::swap(VB, Vg);
    }
    small_gemm(B, 0, VB, 0, S, m, 1.0, 0.0, s);
    small_gemm(VB, 1, S, 0, B, m, 1.0, 0.0, s);    // U^T B U
    small_gemm(W1, 0, VB, 0, W2, m, 1.0, 0.0, s);  // V1 U
    std::swap(W1, W2);
  }
  jacobi_launch<double>(B, m, w, VB, Vg, 40, 1e-17, 1e-32, 8 * DBL_EPSILON, s);
  small_gemm(W1, 0, VB, 0, V, m, 1.0, 0.0, s);  // V1 V_B
}

// ---------------------------------------------------------------------------
// column reductions over rows
// mode 0: out[i] = sum_r X[r][i] Y[r][i];  mode 1: out[i] = sum_r (Y - th_i X)^2
// Block b sums every B-th group of CR_G rows of every column into part[b];
// a second kernel adds the B partial sums of each column in a fixed order, so
// the result does not depend on the order in which blocks run.
// ---------------------------------------------------------------------------
constexpr int CR_G = 6;
__global__ void k_colred(const double* __restrict__ X, const double* __restrict__ Y,
                         const double* __restrict__ th, int64_t n, int m, int ld, int mode,
                         double* part) {
  // blockDim.y row groups of one thread per column, added in order at the end
  __shared__ double sg[CR_G][128];
  const int i = threadIdx.x;
  const bool on = i < m;
  const double t = mode && on ? th[i] : 0.0;
  double acc = 0.0;
  constexpr int U = 4;  // rows whose loads are in flight together
  const int64_t step = (int64_t)gridDim.x * CR_G;
  for (int64_t r0 = (int64_t)blockIdx.x * CR_G + threadIdx.y; on && r0 < n; r0 += U * step) {
    double x[U], y[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int64_t r = r0 + u * step;
      x[u] = r < n ? X[r * ld + i] : 0.0;
      y[u] = r < n ? Y[r * ld + i] : 0.0;
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      if (mode) {
        const double d = y[u] - t * x[u];
        acc = fma(d, d, acc);
      } else {
        acc = fma(x[u], y[u], acc);
      }
    }
  }
  if (on) sg[threadIdx.y][i] = acc;
  __syncthreads();
  if (on && threadIdx.y == 0) {
    for (int g = 1; g < CR_G; ++g) acc += sg[g][i];
    part[(int64_t)blockIdx.x * m + i] = acc;
  }
}

// one warp per column: lane l adds the partials l, l + 32, ... in order, then
// the lanes by a fixed tree
__global__ void __launch_bounds__(32) k_colsum(const double* __restrict__ part, int nparts, int m,
                                               double* out) {
  const int i = blockIdx.x;
  double s = 0.0;
  for (int b = threadIdx.x; b < nparts; b += 32) s += part[(int64_t)b * m + i];
  s = warp_sum(s);
  if (threadIdx.x == 0) out[i] = s;
}

static void colred(const double* X, const double* Y, const double* th, int64_t n, int m, int ld,
                   int mode, double* out, double* part, int num_sms, cudaStream_t s) {
  const int threads = ((m + 31) / 32) * 32;
  RF_CHECK(m <= 128, RAFEAST_ERR_INVALID_ARG);
  const int blocks = (int)std::min<int64_t>((n + CR_G - 1) / CR_G, 2 * (int64_t)num_sms);
  k_colred<<<blocks, dim3(threads, CR_G), 0, s>>>(X, Y, th, n, m, ld, mode, part);
  RF_LAUNCH();
  k_colsum<<<m, 32, 0, s>>>(part, blocks, m, out);
  RF_LAUNCH();
}

void col_dot(const double* X, const double* Y, int64_t n, int m, int ld, double* out,
             double* part, int num_sms, cudaStream_t s) {
  colred(X, Y, nullptr, n, m, ld, 0, out, part, num_sms, s);
}

void col_resid2(const double* Q, const double* AQ, const double* theta, int64_t n, int m, int ld,
                double* out, double* part, int num_sms, cudaStream_t s) {
  colred(Q, AQ, theta, n, m, ld, theta ? 1 : 0, out, part, num_sms, s);
}

// ---------------------------------------------------------------------------
// quadrature combine: Qt = f_i Q + D
// ---------------------------------------------------------------------------
template <typename T>
__global__ void k_combine(const double* __restrict__ Q, int ldq, const T* __restrict__ D, int ldd,
                          const double* __restrict__ f, int64_t n, int m, double* __restrict__ Qt) {
  const int64_t total = n * (int64_t)m;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t r = e / m;
    const int i = (int)(e - r * m);
    Qt[r * ldq + i] = fma(f[i], Q[r * ldq + i], (double)D[r * ldd + i]);
  }
}

template <typename T>
void launch_combine(const double* Q, int ldq, const T* D, int ldd, const double* f, int64_t n,
                    int m, double* Qt, cudaStream_t s) {
  k_combine<T><<<blocks_for(n * (int64_t)m), 256, 0, s>>>(Q, ldq, D, ldd, f, n, m, Qt);
  RF_LAUNCH();
}
template void launch_combine<float>(const double*, int, const float*, int, const double*, int64_t,
                                    int, double*, cudaStream_t);
template void launch_combine<double>(const double*, int, const double*, int, const double*,
                                     int64_t, int, double*, cudaStream_t);

}  // namespace rafeast
