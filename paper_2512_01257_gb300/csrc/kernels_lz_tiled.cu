// Tiled product of the real Lanczos form (float): w = L u_k and the two sums
// of every column (u^T u, u^T w), with the rows cut into tiles (tiling.cpp).
//
// The staging is that of kernels_tiled.cu: a work item is (tile, column
// block); its CTA copies the rows of the tile's union restricted to the
// block's CB chunks of 4 real columns into shared memory with cp.async, then
// every row of the tile gathers its neighbours from there. What bounds it is
// the shared-memory pipe (a 16-byte load per gathered chunk); a real row has
// half the chunks of the complex seed residual. CB divides the row's chunks
// where one of 4, 5, 8, 10 does, so that no lane of a block idles; 8 chunks
// (128 bytes) are free of bank conflicts, the autotuner weighs that against
// the block count.
//
// Sums: float per lane over its rows, FP64 from there on in a fixed order (CTA,
// column block), no atomic addition in a floating-point sum: two runs give the
// same bits. The last CTA of a column block turns them into the block's
// alpha, g, s.
#include <algorithm>

#include "lanczos.cuh"
#include "tiled.cuh"

namespace rafeast {

constexpr int LZ_SUMS = 8;  // sums per chunk: u^T u and u^T w of 4 columns

template <int CB, int MINB, bool VF>
__global__ void __launch_bounds__(TT, MINB) k_lz_dots_tiled(LzArgs<float> a, TileArgs tl) {
  if (__ldcg(&a.ctl->done)) return;
  extern __shared__ __align__(16) P4 xs[];  // [max_union * CB] chunks, a zero row of CB
  __shared__ TileIdx tb;
  __shared__ int sact[CB];
  constexpr int NRS = TT / CB;  // row slots
  const int ncb = tl.ncb;
  const int cbk = blockIdx.x % ncb;
  const int j = threadIdx.x % CB, rs = threadIdx.x / CB;
  const int q = cbk * CB + j;
  if (threadIdx.x < CB) {
    const int qq = cbk * CB + threadIdx.x;
    sact[threadIdx.x] = qq < a.nq ? __ldcg(a.qact + qq) : 0;
  }
  __syncthreads();
  const bool on = rs < NRS && sact[j] != 0;
  int any = 0;
#pragma unroll
  for (int t = 0; t < CB; ++t) any |= sact[t];
  const int64_t ldt = a.ld;
  const int k = __ldcg(&a.dyn->k);
  const float* __restrict__ U = (const float*)__ldcg((const u64*)&a.dyn->du);
  const int32_t* __restrict__ rowptr = VF ? a.lrowptr : a.rowptr;
  u64 du[2] = {0ull, 0ull}, dw[2] = {0ull, 0ull};  // packed float sums
  const int zrow = tl.max_union;
  if (threadIdx.x < CB) xs[zrow * CB + threadIdx.x] = P4{0ull, 0ull};
  const int nitems = tl.ntiles * ncb;
  // the next item's index data travels in registers during this one's gathers
  constexpr int UPT = (TILE_UCAP + TT - 1) / TT, RPT = (TILE_TMAX + 1 + TT - 1) / TT;
  int f_r0 = 0, f_nr = 0, f_nu = 0, f_us = 0;
  int f_sidx[UPT], f_srp[RPT];
  auto fetch = [&](int it) {
    const int t = it / ncb;
    f_r0 = __ldg(tl.trow + t);
    f_nr = __ldg(tl.trow + t + 1) - f_r0;
    const int u0 = __ldg(tl.uoff + t);
    f_nu = __ldg(tl.uoff + t + 1) - u0;
    f_us = __ldg(tl.uself + t);
#pragma unroll
    for (int c = 0; c < UPT; ++c) {
      const int u = threadIdx.x + TT * c;
      f_sidx[c] = u < f_nu ? __ldg(tl.ucol + u0 + u) : 0;
    }
#pragma unroll
    for (int c = 0; c < RPT; ++c) {
      const int r = threadIdx.x + TT * c;
      f_srp[c] = r <= f_nr ? __ldg(rowptr + f_r0 + r) : 0;
    }
  };
  if (any && (int)blockIdx.x < nitems) fetch(blockIdx.x);
  for (int item = blockIdx.x; any && item < nitems; item += gridDim.x) {
    const int r0 = f_r0, nr = f_nr, nu = f_nu;
#pragma unroll
    for (int c = 0; c < UPT; ++c) {
      const int u = threadIdx.x + TT * c;
      if (u < nu) tb.sidx[u] = f_sidx[c];
    }
#pragma unroll
    for (int c = 0; c < RPT; ++c) {
      const int r = threadIdx.x + TT * c;
      if (r <= nr) tb.srp[r] = f_srp[c];
    }
    if (threadIdx.x == 0) {
      tb.r0 = r0;
      tb.nr = nr;
      tb.nu = nu;
      tb.us = f_us;
      tb.kbase = f_srp[0] & ~7;
    }
    __syncthreads();
    tile_copies<CB>(tl, tb, xs, U, ldt, cbk, sact);
    cp_async_wait_all();
    __syncthreads();
    if (item + (int)gridDim.x < nitems) fetch(item + gridDim.x);
    const uint16_t* slx = tb.slx;
    const int kbase = tb.kbase, us = tb.us;
    if (on) {
      for (int lr = rs; lr < nr; lr += NRS) {
        const int64_t row = r0 + lr;
        const int k0 = tb.srp[lr] - kbase, k1 = tb.srp[lr + 1] - kbase;
        // eight entries in flight; entries past the row's end read the zero row
        P4 acc = {0ull, 0ull};
        for (int kk = k0; kk < k1; kk += 8) {
          int id[8];
#pragma unroll
          for (int e = 0; e < 8; ++e) id[e] = kk + e < k1 ? (int)slx[kk + e] : zrow;
          P4 x[8];
#pragma unroll
          for (int e = 0; e < 8; ++e) x[e] = xs[id[e] * CB + j];
          if constexpr (VF) {
#pragma unroll
            for (int e = 0; e < 8; ++e) acc = p4add(acc, x[e]);
          } else {
            const float* v = a.val + kbase + kk;
            float vv[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) vv[e] = kk + e < k1 ? __ldg(v + e) : 0.0f;
#pragma unroll
            for (int e = 0; e < 8; ++e) acc = p4fma(splat2(vv[e]), x[e], acc);
          }
        }
        const P4 uv = xs[(us + lr) * CB + j];
        P4 w = acc;
        if constexpr (VF) {  // L u = deg u - (sum over neighbours)
          const u64 deg = splat2((float)(k1 - k0)), m1 = splat2(-1.0f);
          w = P4{fma2(deg, uv.lo, fma2(m1, acc.lo, 0ull)), fma2(deg, uv.hi, fma2(m1, acc.hi, 0ull))};
        }
        du[0] = fma2(uv.lo, uv.lo, du[0]);
        du[1] = fma2(uv.hi, uv.hi, du[1]);
        dw[0] = fma2(uv.lo, w.lo, dw[0]);
        dw[1] = fma2(uv.hi, w.hi, dw[1]);
        *reinterpret_cast<P4*>(a.w + row * ldt + (int64_t)q * 4) = w;
      }
    }
    __syncthreads();  // the next item's copies overwrite the staged data
  }
  // CTA sums in a fixed order: the row slots of each chunk position in turn
  double* sred = reinterpret_cast<double*>(xs);  // [NRS][CB][LZ_SUMS]
  if (rs < NRS) {
    double* o = sred + (rs * CB + j) * LZ_SUMS;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const float2 x = lo2(du[h]), y = lo2(dw[h]);
      o[4 * h + 0] = (double)x.x;
      o[4 * h + 1] = (double)y.x;
      o[4 * h + 2] = (double)x.y;
      o[4 * h + 3] = (double)y.y;
    }
  }
  __syncthreads();
  if (threadIdx.x < CB * LZ_SUMS) {
    double s = 0.0;
    for (int r = 0; r < NRS; ++r) s += sred[r * CB * LZ_SUMS + threadIdx.x];
    tl.part[(int64_t)blockIdx.x * CB * LZ_SUMS + threadIdx.x] = s;
    __threadfence();
  }
  __syncthreads();
  const int per_block = (int)gridDim.x / ncb;
  __shared__ int s_last;
  if (threadIdx.x == 0) s_last = atomicAdd(&a.ctl->cbticket[cbk], 1u) == (unsigned)per_block - 1;
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  double* s_acc = reinterpret_cast<double*>(xs);  // [CB * LZ_SUMS]: 2 per column
  {
    // lane l adds the CTAs l, l + 32, ... of the block, then the warp adds its
    // lanes by a fixed tree; a warp takes the sums warp, warp + TT/32, ...
    constexpr int NW = TT / 32, VPW = (CB * LZ_SUMS + NW - 1) / NW;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    double sv[VPW];
#pragma unroll
    for (int u = 0; u < VPW; ++u) sv[u] = 0.0;
    for (int b0 = 0; b0 < per_block; b0 += 32) {
      const int b = b0 + lane;
      double pv[VPW];
#pragma unroll
      for (int u = 0; u < VPW; ++u) {
        const int v = warp + NW * u;
        pv[u] = (v < CB * LZ_SUMS && b < per_block)
                    ? __ldcg(tl.part + (int64_t)(cbk + b * ncb) * CB * LZ_SUMS + v)
                    : 0.0;
      }
      if (b < per_block) {
#pragma unroll
        for (int u = 0; u < VPW; ++u) sv[u] += pv[u];
      }
    }
#pragma unroll
    for (int u = 0; u < VPW; ++u) {
      const int v = warp + NW * u;
      double x = sv[u];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
      if (lane == 0 && v < CB * LZ_SUMS) s_acc[v] = x;
    }
  }
  __syncthreads();
  if (!a.dry)  // (dry: a timing run)
    lz_column_scalars<float>(a, k, 4 * cbk * CB, 4 * min(a.nq, cbk * CB + CB), s_acc);
  if (threadIdx.x != 0) return;
  // the last column block to finish ends the step
  CocgCtl* c = a.ctl;
  c->cbticket[cbk] = 0;
  __threadfence();
  if (atomicAdd(&c->ticket, 1u) != (unsigned)ncb - 1) return;
  c->ticket = 0;
  if (!a.dry) lz_advance<float>(a, k);
  __threadfence();
}

template <int CB, int MINB, bool VF>
static void launch_cb(const LzArgs<float>& a, const TileArgs& tl, int num_sms, int occ_cap,
                      cudaStream_t s) {
  auto kern = k_lz_dots_tiled<CB, MINB, VF>;
  const size_t stage = (size_t)(tl.max_union + 1) * CB * sizeof(P4);
  const size_t red = (size_t)(TT / CB) * CB * LZ_SUMS * sizeof(double);
  const size_t smem = std::max(stage, red);
  ensure_dyn_smem(reinterpret_cast<const void*>(kern), smem);
  int occ = 0;
  RF_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, TT, smem));
  occ = std::min(std::max(occ, 1), TILE_MAX_OCC);  // tl.part holds num_sms * TILE_MAX_OCC CTAs
  if (occ_cap > 0 && occ > occ_cap) occ = occ_cap;
  const int g = std::max((num_sms * occ / tl.ncb) * tl.ncb, tl.ncb);
  kern<<<g, TT, smem, s>>>(a, tl);
  RF_LAUNCH();
}

void launch_lz_dots_tiled(const LzArgs<float>& a, const TileArgs& tl, int num_sms, int occ_cap,
                          cudaStream_t s) {
  const bool vf = a.lcolidx != nullptr;
  switch (tl.cb) {
    case 4: vf ? launch_cb<4, 4, true>(a, tl, num_sms, occ_cap, s)
               : launch_cb<4, 4, false>(a, tl, num_sms, occ_cap, s); break;
    case 5: vf ? launch_cb<5, 4, true>(a, tl, num_sms, occ_cap, s)
               : launch_cb<5, 4, false>(a, tl, num_sms, occ_cap, s); break;
    case 8: vf ? launch_cb<8, 3, true>(a, tl, num_sms, occ_cap, s)
               : launch_cb<8, 3, false>(a, tl, num_sms, occ_cap, s); break;
    case 10: vf ? launch_cb<10, 2, true>(a, tl, num_sms, occ_cap, s)
                : launch_cb<10, 2, false>(a, tl, num_sms, occ_cap, s); break;
    default: throw Err{RAFEAST_ERR_INVALID_ARG};
  }
}

}  // namespace rafeast
