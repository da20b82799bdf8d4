// Kernels of the real Lanczos form of the multi-shift solve, one problem per
// launch (recurrences, data layout and bodies: lanczos.cuh).
#include <algorithm>

#include "lanczos.cuh"

namespace rafeast {

// u_0 = b (0 in a padding column), D = 0, and the scalars of every column and
// node; q/aq hold m columns of stride ldq
template <typename T>
__global__ void __launch_bounds__(THREADS) k_lz_init(LzArgs<T> a, const double* __restrict__ q,
                                                     const double* __restrict__ aq,
                                                     const double* __restrict__ theta, int ldq,
                                                     int m, int form) {
  const int64_t total = a.n * (int64_t)a.ld;
  T* u = (T*)a.dyn->slab[0];
  const int64_t t0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int64_t st = (int64_t)gridDim.x * blockDim.x;
  for (int64_t e = t0; e < total; e += st) {
    const int64_t row = e / a.ld;
    const int c = (int)(e - row * a.ld);
    double b = 0.0;
    if (c < m) {
      b = q[row * ldq + c];
      if (form == RAFEAST_FORM_CORRECTION) b = aq[row * ldq + c] - theta[c] * b;
    }
    u[e] = (T)b;
    a.dacc[e] = (T)0;
  }
  for (int64_t c = t0; c < a.ld; c += st) {
    LzCol x;
    x.rr = x.irr = x.s = x.is = x.sq = 1.0;
    x.bnorm2 = 0.0;
    x.bad = 0;
    x.kstop = LZ_RUNS;
    a.col[c] = x;
    for (int t = 0; t < 3; ++t) a.acc[3 * c + t] = 0.0;
    if (c < a.nq) a.qact[c] = 1;
  }
  for (int64_t e = t0; e < (int64_t)a.ld * a.nc; e += st) {
    LzShift x;
    x.rho = make_double2(1.0, 0.0);
    x.dinv = make_double2(0.0, 0.0);
    x.kstop = LZ_RUNS;
    x.pad = 0;
    a.sh[e] = x;
  }
  if (t0 == 0) {
    CocgCtl c = {};
    c.g_mn = 0x7fffffff;
    c.active = a.ld;
    *a.ctl = c;
    a.dyn->k = 0;
    a.dyn->du = a.dyn->slab[0];
  }
}

template <typename T, int MAXCPL, int MINB, bool VF, bool FX = false, bool SQ = FX>
__global__ void __launch_bounds__(THREADS, MINB) k_lz_dots(LzArgs<T> a) {
  constexpr int NBX = !FX ? 0 : MAXCPL == 1 && MINB > 3 ? 4 : MAXCPL == 2 && MINB > 2 ? 2 : 0;
  lz_dots_body<T, MAXCPL, VF, FX, SQ, NBX>(a, grid_blk());
}

template <typename T, bool FX>
__global__ void __launch_bounds__(THREADS) k_lz_update(LzArgs<T> a, int sb) {
  // (a CTA with a share of the scalars cannot see `done` set by this step: it
  // waits for every share; the others have no barrier below)
  if (__ldcg(&a.ctl->done)) return;
  if ((int)blockIdx.x < sb) {
    lz_scalar_share<T>(a, __ldcg(&a.dyn->k) - 1, blockIdx.x, sb);
    return;
  }
  // contiguous row ranges, the first CTA's at the top
  const int64_t nb = gridDim.x - sb, per = (a.n + nb - 1) / nb;
  const int64_t r1 = a.n - (int64_t)(blockIdx.x - sb) * per;
  if (r1 > 0) lz_update_rows<T, FX>(a, r1 > per ? r1 - per : 0, r1);
}

template <typename T>
__global__ void __launch_bounds__(32) k_lz_comp(LzArgs<T> a, int k0, int k1, int dirs) {
  __shared__ double tile[32][17];
  __shared__ LzRing ring;
  const int cap = lz_stage_ring(a, ring);
  lz_comp_col<T>(a, ring, cap, blockIdx.x, k0, k1, dirs != 0, tile);
}

template <typename T>
__global__ void __launch_bounds__(THREADS, 2) k_lz_sum(LzArgs<T> a, int k0, int k1) {
  __shared__ LzRing ring;
  const int cap = lz_stage_ring(a, ring);
  const int64_t per = (a.n + gridDim.x - 1) / gridDim.x, r0 = (int64_t)blockIdx.x * per;
  lz_sum_rows<T>(a, ring, cap, k0, k1, r0, r0 + per < a.n ? r0 + per : a.n);
}

template <typename T, int JB, int RPT>
__global__ void __launch_bounds__(THREADS, 2) k_lz_apply(LzArgs<T> a, int j0, int k0, int k1) {
  __shared__ LzRing ring;
  const int cap = lz_stage_ring(a, ring);
  const int64_t per = (a.n + gridDim.x - 1) / gridDim.x, r0 = (int64_t)blockIdx.x * per;
  lz_apply_rows<T, JB, RPT>(a, ring, cap, j0, k0, k1, r0, r0 + per < a.n ? r0 + per : a.n);
}

template <typename T>
void launch_lz_init(const LzArgs<T>& a, const double* q, const double* aq, const double* theta,
                    int ldq, int m, int form, int num_sms, cudaStream_t s) {
  const int64_t total = a.n * (int64_t)a.ld;
  int64_t blocks = std::min<int64_t>((total + THREADS - 1) / THREADS, (int64_t)num_sms * 8);
  k_lz_init<T><<<(int)std::max<int64_t>(blocks, 1), THREADS, 0, s>>>(a, q, aq, theta, ldq, m, form);
  RF_LAUNCH();
}

template <typename T, int MAXCPL, int MINB>
static void dots_inst(const LzArgs<T>& a, LzSums sums, int num_sms, cudaStream_t s) {
  RF_CHECK(a.cpl <= MAXCPL && (sums == LZ_PLAIN || (sizeof(T) == 8 && a.lcolidx && a.qe)),
           RAFEAST_ERR_INVALID_ARG);
  auto kern = a.lcolidx ? k_lz_dots<T, MAXCPL, MINB, true> : k_lz_dots<T, MAXCPL, MINB, false>;
  if constexpr (sizeof(T) == 8) {
    if (sums == LZ_FIX) kern = k_lz_dots<T, MAXCPL, MINB, true, true>;
    else if (sums == LZ_SQ) kern = k_lz_dots<T, MAXCPL, MINB, true, false, true>;
  }
  const size_t smem = lz_dots_smem<T>(a.lanes, MAXCPL, a.ld, sums == LZ_PLAIN ? 2 : 3);
  if (smem > 48 * 1024) ensure_dyn_smem(reinterpret_cast<const void*>(kern), smem);
  const int colblocks = (a.nq + a.lanes * a.cpl - 1) / (a.lanes * a.cpl);
  const int64_t per = (int64_t)WARPS * (32 / a.lanes);
  dim3 grid(grid_x(kern, smem, num_sms, (a.n + per - 1) / per), colblocks);
  kern<<<grid, THREADS, smem, s>>>(a);
  RF_LAUNCH();
}

// occ: CTAs per SM the instance is compiled for (0: the default of its width);
// sums: LZ_FIX gathers from the fixed-point copy of u_k (a.qu, k > 0), LZ_SQ is
// the step before the first of those
template <typename T>
void launch_lz_dots(const LzArgs<T>& a, LzSums sums, int occ, int num_sms, cudaStream_t s) {
  RF_CHECK(a.lanes > 0 && a.cpl > 0, RAFEAST_ERR_INVALID_ARG);
  if (a.cpl == 1) {
    if (occ == 3) dots_inst<T, 1, 3>(a, sums, num_sms, s);
    else dots_inst<T, 1, 4>(a, sums, num_sms, s);
  } else if (a.cpl == 2) {
    if (occ == 2) dots_inst<T, 2, 2>(a, sums, num_sms, s);
    else dots_inst<T, 2, 3>(a, sums, num_sms, s);
  } else {
    dots_inst<T, 4, 2>(a, sums, num_sms, s);
  }
}

template <typename T>
void launch_lz_update(const LzArgs<T>& a, int num_sms, cudaStream_t s) {
  RF_CHECK(a.nq <= THREADS && a.nc <= 16, RAFEAST_ERR_INVALID_ARG);
  const int per = THREADS / a.nq;
  // the scalars, two columns (a warp each) to a CTA of its own ahead of the rows: their
  // latency chain runs beside the streaming, not before the rows of the same CTA
  // (40 x 50 grid, 24 columns, FP64: a step 23.2 -> 20.8 us; kNN graph of 8,000 rows, 42
  // columns: 48 -> 45 us with its share of the solve. Eight columns a CTA, whose warps
  // share one FP64 pipe: 23.9 us on the grid)
  const int sb = (a.ld + 1) / 2;
  const int64_t blocks =
      sb + std::min<int64_t>((a.n + per - 1) / per, std::max(num_sms * 6 - sb, 1));
  if constexpr (sizeof(T) == 8) {
    if (a.qu) k_lz_update<T, true><<<(int)blocks, THREADS, 0, s>>>(a, sb);
    else k_lz_update<T, false><<<(int)blocks, THREADS, 0, s>>>(a, sb);
  } else {
    k_lz_update<T, false><<<(int)blocks, THREADS, 0, s>>>(a, sb);
  }
  RF_LAUNCH();
}

template <typename T, int JB, int RPT>
static void apply_inst(const LzArgs<T>& a, int j0, int k0, int k1, int num_sms, cudaStream_t s) {
  const int64_t per = (int64_t)(THREADS / a.nq) * RPT;
  const int64_t gx = std::min<int64_t>((int64_t)num_sms * 2, (a.n + per - 1) / per);
  k_lz_apply<T, JB, RPT><<<(int)gx, THREADS, 0, s>>>(a, j0, k0, k1);
  RF_LAUNCH();
}

template <typename T>
void launch_lz_collapse(const LzArgs<T>& a, int k0, int k1, bool last, int num_sms,
                        cudaStream_t s) {
  if (k1 <= k0) return;
  const bool dirs = !last || k0 > 0;
  k_lz_comp<T><<<a.ld, 32, 0, s>>>(a, k0, k1, dirs ? 1 : 0);
  RF_LAUNCH();
  if (!dirs) {
    const int64_t per = (int64_t)(THREADS / a.nq) * 4;
    const int64_t gx = std::min<int64_t>((int64_t)num_sms * 2, (a.n + per - 1) / per);
    k_lz_sum<T><<<(int)gx, THREADS, 0, s>>>(a, k0, k1);
    RF_LAUNCH();
    return;
  }
  // nodes in passes of at most 4
  if (a.nc <= 1) apply_inst<T, 1, 4>(a, 0, k0, k1, num_sms, s);
  else if (a.nc <= 2) apply_inst<T, 2, 2>(a, 0, k0, k1, num_sms, s);
  else
    for (int j0 = 0; j0 < a.nc; j0 += 4)
      apply_inst<T, 4, sizeof(T) == 4 ? 1 : 2>(a, j0, k0, k1, num_sms, s);
}

#define LZ_INST(T)                                                                             \
  template void launch_lz_init<T>(const LzArgs<T>&, const double*, const double*,              \
                                  const double*, int, int, int, int, cudaStream_t);            \
  template void launch_lz_dots<T>(const LzArgs<T>&, LzSums, int, int, cudaStream_t);             \
  template void launch_lz_update<T>(const LzArgs<T>&, int, cudaStream_t);                      \
  template void launch_lz_collapse<T>(const LzArgs<T>&, int, int, bool, int, cudaStream_t);
LZ_INST(float)
LZ_INST(double)

}  // namespace rafeast
