// Multi-shift solve of (z_j I - A) X_j = B over a real Lanczos recurrence.
//
// B and A are real, so the Krylov space of every shift and column is real: the
// conjugate-orthogonal-CG residual of shift j after k steps is a complex
// number times the Lanczos vector u_k of the column. One real recurrence per
// column
//     u_{k+1} = s_k (L u_k - alpha_k u_k - g_k u_{k-1}),
//     alpha_k = u_k^T L u_k / rr_k,  rr_k = u_k^T u_k,
//     g_k = rr_k / (s_{k-1} rr_{k-1}),   u_0 = b,
// therefore serves every node (Lanczos 1950; the scaling s_k keeps ||u_k||
// near ||b|| and is part of the recurrence, so it costs no accuracy), and the
// COCG iterates of node z (shift sigma of A taken off) follow from the LDL^T
// factors of the tridiagonal z - T:
//     q_k = u_k + t_k q_{k-1},        t_k = g_k / delta_{k-1},
//     delta_k = z - alpha_k - t_k / s_{k-1},
//     x_{k+1} = x_k + eta_k q_k,      eta_k = rho_k / delta_k,
//     r_{k+1} = rho_{k+1} u_{k+1},    rho_{k+1} = eta_k / s_k,  rho_0 = 1.
// Im(delta_k) never vanishes for Im(z) > 0, so no pivot breaks down.
//
// Neither x_j nor the directions q_j are kept step by step: every u_k stays in a
// slot of a ring that grows with the solve, t_k and w_j eta_k beside it. When
// the solve ends, the recurrences of all its steps are collapsed, backwards,
// into one real coefficient per step and column (k_lz_comp),
//     D = sum_k c_k u_k,   c_k = Re sum_j e_jk,  e_jk = w_j eta_jk + t_j,k+1 e_j,k+1,
// and one pass over the ring forms D (k_lz_sum). A step then moves 7 real
// values per row and column (the product reads u and writes w = L u, the
// update reads u, w, u_{k-1} and writes u_{k+1}, the pass reads u), against 32
// for the complex seed recurrence with three stored shifted directions
// (kernels_sparse.cu). On the kNN graph of 200,000 rows and 80 columns (N_c = 4,
// float) a step took 0.16 + 0.33 ms (product, update) and takes 0.092 + 0.061
// ms; on the million-row grid with 96 columns 0.55 + 1.4 ms became 0.26 + 0.31
// ms. A ring that may not grow further (memory) is taken up
// when it is full: the chunk's steps go into D and into the directions
//     p_j = a_j p_j + sum_k b_jk u_k,   D += Re sum_j g_j p_j   (k_lz_apply),
// and the next chunk reuses the slots.
//
// The scalar work is spread out, because one SM issues FP64 at 1/64 of the
// float rate: the last CTA of the product turns the sums into alpha, g, s (one
// reciprocal per column), and the update kernel's CTAs advance delta, rho and
// the stopping rule of a column or two each, beside their streaming.
//
// Rows hold ld real values (a multiple of 4); a lane owns 16-byte chunks: 4
// columns in float, 2 in double. In float the coefficients alpha, g, s are
// rounded to float before the scalar recurrences use them, so the tridiagonal
// matrix is exactly the one the vectors were made with.
#pragma once

#include "cocg_kernels.cuh"

namespace rafeast {

template <typename T> constexpr int LZV = 16 / (int)sizeof(T);  // columns per chunk
template <typename T> struct LzVec {
  using t = typename std::conditional<sizeof(T) == 4, float4, double2>::type;
};
__device__ __forceinline__ void lz_get(const float4& x, float (&v)[4]) {
  v[0] = x.x; v[1] = x.y; v[2] = x.z; v[3] = x.w;
}
__device__ __forceinline__ void lz_get(const double2& x, double (&v)[2]) { v[0] = x.x; v[1] = x.y; }
__device__ __forceinline__ float4 lz_put(const float (&v)[4]) { return make_float4(v[0], v[1], v[2], v[3]); }
__device__ __forceinline__ double2 lz_put(const double (&v)[2]) { return make_double2(v[0], v[1]); }

// address of slot k of the ring
template <typename T>
__device__ __forceinline__ char* lz_slot(const LzArgs<T>& a, int k) {
  const int s = k % __ldcg(&a.dyn->cap);
  return (char*)__ldcg((const unsigned long long*)&a.dyn->slab[s / a.sl]) +
         (int64_t)(s % a.sl) * a.stride;
}
// the same through a copy of the slab table in shared memory
struct LzRing {
  char* slab[LZ_SLABS];
};
template <typename T>
__device__ __forceinline__ int lz_stage_ring(const LzArgs<T>& a, LzRing& ring) {
  const int cap = __ldcg(&a.dyn->cap), n = (cap + a.sl - 1) / a.sl;
  for (int t = threadIdx.x; t < n; t += blockDim.x)
    ring.slab[t] = (char*)__ldcg((const unsigned long long*)&a.dyn->slab[t]);
  __syncthreads();
  return cap;
}
template <typename T>
__device__ __forceinline__ char* lz_slot(const LzArgs<T>& a, const LzRing& ring, int cap, int k) {
  const int s = k % cap;
  return ring.slab[s / a.sl] + (int64_t)(s % a.sl) * a.stride;
}
template <typename T>
__device__ __forceinline__ double2* lz_th(const LzArgs<T>& a, char* slot) {
  return reinterpret_cast<double2*>(slot + a.uoff);
}

// Fixed-point neighbour sums (double, LzArgs::qu). FP64 adds issue at 1/64 of
// the integer rate on this chip, so a neighbour sum of a unit-weight Laplacian
// is formed in 64-bit integers: the update leaves u_{k+1} a second time as
// rint(u 2^-E) with one E per column, the product adds those (exactly, modulo
// 2^64) and returns to FP64 once per row. E is the least exponent for which no
// sum can leave the range whatever the vector: with N_i the neighbours of i,
//     |sum_{N_i} u| <= sqrt(max degree) ||u_{k+1}||,
//     ||u_{k+1}|| <= s (||w - alpha u_k|| + g ||u_{k-1}||),
// the first norm from the sums u^T u, u^T w, w^T w of the product (a slack of
// 2^-30 w^T w covers their rounding; it counts where w is alpha u_k to 2^-15,
// and is then 2^-15 ||w|| against the 2^-53 ||w|| that w itself is rounded by,
// far above 2^-62 of the slack). The rounding to units of 2^E is an error of
// the next w; filter_lz_run takes this path where it stays below the rounding
// of w - alpha u_k, which u_{k+1} carries anyway. Geometric graph of 16,000 rows (68
// neighbours, 69 columns): a step of the FP64 filter 218 -> 89 us, product 73 us of it.
// False where the bound leaves the double range (its w^T w does from a norm of
// about 1e152 on, before the sums of the recurrence do): no unit is safe then.
template <typename T>
__device__ __forceinline__ bool lz_fix_exponent(const LzArgs<T>& a, double rr, double ul, double ww,
                                                double alpha, double g, double s, double rr_prev,
                                                int& E) {
  const double au = alpha * ul;  // (at most w^T w)
  const double t2 = fmax(ww - au - alpha * (ul - alpha * rr), 0.0) + 0x1p-30 * ww;
  const double x = a.rootdeg * 1.001 * s * (sqrt(t2) + g * sqrt(rr_prev));
  E = 0;
  if (!isfinite(x) || !isfinite(au)) return false;
  if (x > 0.0) E = max(-900, min(900, ilogb(x) + 1 - 63));
  return true;
}
// rint(y 2^-E), ties away from zero, in integer arithmetic (FP64 conversions
// and products would cost more than the sum they prepare)
__device__ __forceinline__ long long lz_fix(double y, int E) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(y);
  const int sh = (int)((b >> 52) & 0x7ff) - 1075 - E;  // (a subnormal y is below every unit)
  unsigned long long m = (b & 0xfffffffffffffull) | 0x10000000000000ull;
  if (sh >= 0) {
    m <<= min(sh, 11);  // (11 at most: more means a column of infinities or NaN, which has stopped)
  } else {
    const int r = min(-sh, 63);
    m = (m + (1ull << (r - 1))) >> r;
  }
  return (long long)b < 0 ? -(long long)m : (long long)m;
}

// alpha, g, s of the columns [c0, c1) at step k from their NS sums (rr,
// u^T L u and, of three, w^T w at sums[NS (c - c0)], any address space), by
// the CTA that ends the product
template <typename T, int NS = 2>
__device__ void lz_column_scalars(const LzArgs<T>& a, int k, int c0, int c1, const double* sums) {
  for (int c = c0 + (int)threadIdx.x; c < c1; c += blockDim.x) {
    LzCol& st = a.col[c];
    LzCoef<T> cf;
    cf.alpha = cf.g = cf.s = cf.pad = (T)0;
    int E = 0;
    bool unit = true;
    if (st.kstop == LZ_RUNS) {
      const double rr = sums[NS * (c - c0)], ul = sums[NS * (c - c0) + 1];
      const double irr = 1.0 / rr, irr_prev = st.irr;
      if (k == 0) st.bnorm2 = rr;
      if (rr > 0.0) {
        cf.alpha = (T)(ul * irr);
        if (k > 0) {
          cf.g = (T)(rr * irr_prev * st.is);
          cf.s = (T)(st.s * st.sq * irr);  // s_{k-1} sqrt(||b||^2 rr_{k-1}) / rr_k
        } else {
          cf.s = cf.alpha != (T)0 ? (T)(1.0 / fabs((double)cf.alpha)) : (T)1;
        }
      }
      if constexpr (NS == 3)
        unit = lz_fix_exponent(a, rr, ul, sums[NS * (c - c0) + 2], (double)cf.alpha, (double)cf.g,
                               (double)cf.s, st.rr, E);
      st.rr = rr;
      st.irr = irr;
      st.bad = !unit || !isfinite(rr) || !isfinite(ul) || !isfinite((double)cf.alpha) ||
               !isfinite((double)cf.g) || !isfinite((double)cf.s) || (rr > 0.0 && !(cf.s > (T)0));
      // the column stops at this step, broken down or converged (an eigenvector's
      // last scale can leave the range): its next vector is 0, for an infinite one
      // would meet a coefficient of 0 in the sum over the ring
      if (st.bad) {
        cf.alpha = cf.g = cf.s = (T)0;
        E = 0;
      }
    }
    a.cf[c] = cf;
    if constexpr (NS == 3) a.qe[c] = E;
  }
}

// the product's end (one thread): the slots of this step's update and of the
// next product, the step counter
template <typename T>
__device__ void lz_advance(const LzArgs<T>& a, int k) {
  LzDyn* d = a.dyn;
  d->uu = d->du;
  d->up = k > 0 ? lz_slot(a, k - 1) : nullptr;
  d->un = lz_slot(a, k + 1);
  d->du = d->un;
  d->k = k + 1;
  __threadfence();
}

// one column's nodes at step k (one warp; lane j has node j): t_k, delta_k,
// eta_k, rho_{k+1}, the stopping rule; counters by lane 0 into cnt
template <typename T>
__device__ __forceinline__ void lz_nodes(const LzArgs<T>& a, int k, int c, double2* th,
                                         MsCount& cnt) {
  const int j = threadIdx.x & 31, nc = a.nc;
  const LzCol st = a.col[c];
  if (st.kstop != LZ_RUNS) return;
  const double alpha = (double)a.cf[c].alpha, g = (double)a.cf[c].g, s = (double)a.cf[c].s;
  const double is = 1.0 / s, thr = stop_threshold(a.tol2, st.bnorm2);
  bool run = false, conv = false, brk = false, was = false;
  double worst = 0.0;
  if (j < nc) {
    const int64_t sys = (int64_t)c * nc + j;
    LzShift ss = a.sh[sys];
    double2 t = make_double2(0.0, 0.0), ce = t;
    was = ss.kstop == LZ_RUNS;
    if (was) {
      const double nu = (ss.rho.x * ss.rho.x + ss.rho.y * ss.rho.y) * st.rr;
      if (st.bnorm2 > 0.0) worst = nu / st.bnorm2;
      conv = nu <= thr;
      run = !conv && k < a.max_inner && !st.bad;
      if (run) {
        const double2 z = a.z[j], w = a.coef[sys];
        t = make_double2(g * ss.dinv.x, g * ss.dinv.y);
        const double dr = z.x - alpha - t.x * st.is, di = z.y - t.y * st.is;
        const double id = 1.0 / (dr * dr + di * di);
        ss.dinv = make_double2(dr * id, -di * id);
        const double2 eta = make_double2(ss.rho.x * ss.dinv.x - ss.rho.y * ss.dinv.y,
                                         ss.rho.x * ss.dinv.y + ss.rho.y * ss.dinv.x);
        brk = !isfinite(eta.x) || !isfinite(eta.y);
        run = !brk;
        ce = make_double2(w.x * eta.x - w.y * eta.y, w.x * eta.y + w.y * eta.x);
        ss.rho = make_double2(eta.x * is, eta.y * is);
      } else {
        brk = !conv && st.bad;
      }
      if (!run) {
        t = ce = make_double2(0.0, 0.0);
        ss.kstop = k;
      }
      a.sh[sys] = ss;
    }
    th[2 * sys] = t;
    th[2 * sys + 1] = ce;
  }
  const unsigned m = 0xffffffffu;
  const bool any = __any_sync(m, run);
  const int nstop = __popc(__ballot_sync(m, was && !run));
  const int nbrk = __popc(__ballot_sync(m, brk));
  const int ncap = __popc(__ballot_sync(m, was && !run && !conv && !brk));
  if (a.hist)
    for (int o = 16; o > 0; o >>= 1) worst = fmax(worst, __shfl_xor_sync(m, worst, o));
  if (j == 0) {
    cnt.brk += nbrk;
    cnt.cap += ncap;
    if (nstop && st.bnorm2 > 0.0) {
      cnt.mx = max(cnt.mx, k);
      cnt.mn = min(cnt.mn, k);
    }
    cnt.worst = fmax(cnt.worst, worst);
    LzCol& o = a.col[c];
    if (any) {
      o.s = s;
      o.is = is;
      o.sq = sqrt(st.bnorm2) * sqrt(st.rr);  // (their product may leave the range)
      ++cnt.active;
    } else {
      o.kstop = k;
    }
  }
}

// the scalar share of CTA b of nb: warp w takes the columns b + nb w,
// + 8 nb, ...; every CTA with a share (b < nb) calls it with all its threads. The last of them ends the step.
template <typename T>
__device__ __forceinline__ void lz_scalar_share(const LzArgs<T>& a, int k, int b, int nb) {
  if (b >= nb) return;
  constexpr int V = LZV<T>;
  __shared__ MsCount sc[WARPS];
  __shared__ int s_end;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  MsCount cnt;
  ms_count_init(cnt);
  double2* th = lz_th(a, (char*)__ldcg((const unsigned long long*)&a.dyn->uu));
  for (int c = b + nb * warp; c < a.ld; c += nb * WARPS) lz_nodes<T>(a, k, c, th, cnt);
  if (lane == 0) sc[warp] = cnt;
  __syncthreads();
  CocgCtl* ctl = a.ctl;
  if (threadIdx.x == 0) {
    for (int w = 1; w < WARPS; ++w) {
      cnt.active += sc[w].active;
      cnt.brk += sc[w].brk;
      cnt.cap += sc[w].cap;
      cnt.mx = max(cnt.mx, sc[w].mx);
      cnt.mn = min(cnt.mn, sc[w].mn);
      cnt.worst = fmax(cnt.worst, sc[w].worst);
    }
    if (cnt.active) atomicAdd(&ctl->g_active, cnt.active);
    if (cnt.brk) atomicAdd(&ctl->g_brk, cnt.brk);
    if (cnt.cap) atomicAdd(&ctl->g_cap, cnt.cap);
    if (cnt.mx) atomicMax(&ctl->g_mx, cnt.mx);
    if (cnt.mn != 0x7fffffff) atomicMin(&ctl->g_mn, cnt.mn);
    if (a.hist) atomicMax(&ctl->g_worst, (unsigned long long)__double_as_longlong(cnt.worst));
    __threadfence();
    s_end = atomicAdd(&ctl->ticket2, 1u) == (unsigned)nb - 1;
  }
  __syncthreads();
  if (!s_end || warp != 0) return;
  __threadfence();
  for (int q = lane; q < a.nq; q += 32) {
    int any = 0;
#pragma unroll
    for (int v = 0; v < V; ++v) any |= __ldcg(&a.col[q * V + v].kstop) == LZ_RUNS;
    a.qact[q] = any;
  }
  __syncwarp();
  if (lane == 0) {
    const int act = __ldcg(&ctl->g_active), mx = __ldcg(&ctl->g_mx), mn = __ldcg(&ctl->g_mn);
    if (a.hist && k <= a.max_inner) {
      a.hist[k] = act;
      a.rhist[k] = sqrt(__longlong_as_double((long long)__ldcg(&ctl->g_worst)));
    }
    ctl->active = act;
    ctl->breakdown += __ldcg(&ctl->g_brk);
    ctl->capped += __ldcg(&ctl->g_cap);
    if (mx > ctl->max_iters) ctl->max_iters = mx;
    if (mn != 0x7fffffff && (ctl->min_iters == 0 || mn < ctl->min_iters)) ctl->min_iters = mn;
    ctl->iter = k + 1;
    ctl->g_active = ctl->g_brk = ctl->g_cap = ctl->g_mx = 0;
    ctl->g_mn = 0x7fffffff;
    ctl->g_worst = 0ull;
    ctl->ticket2 = 0;
    __threadfence();
    if (act == 0) ctl->done = 1;
    __threadfence();
  }
}

// ---------------------------------------------------------------------------
// product with register gathers: w = L u and the two sums of every column.
// The lane mapping and gather core of cocg_kernels.cuh, a 16-byte chunk of
// real columns in the place of a chunk of complex shifts. What bounds it: the
// latency of the gathers in L1/L2 (float), the FP64 pipe (double).
// ---------------------------------------------------------------------------
// the gather core over the fixed-point copy: NB entries in flight, sums modulo
// 2^64 in any order are the same
template <int MAXCPL, int NB>
__device__ __forceinline__ void gather_row_fix(const int32_t* __restrict__ colidx, int k0, int k1,
                                               int row, int lg, int G, unsigned gmask,
                                               const long long* __restrict__ X, int64_t ld,
                                               const int (&coff)[MAXCPL], unsigned mask,
                                               long long (&acc)[MAXCPL][2]) {
  for (int kb = k0; kb < k1; kb += G) {
    const int my_c = kb + lg < k1 ? __ldg(colidx + kb + lg) : row;
    const int cnt = min(G, k1 - kb);
    for (int e = 0; e < cnt; e += NB) {
      int ci[NB];
#pragma unroll
      for (int u = 0; u < NB; ++u) ci[u] = __shfl_sync(gmask, my_c, e + u < cnt ? e + u : e, G);
      longlong2 x[NB][MAXCPL];
#pragma unroll
      for (int c = 0; c < MAXCPL; ++c)
        if (mask & (1u << c)) {
#pragma unroll
          for (int u = 0; u < NB; ++u)
            x[u][c] = __ldg(reinterpret_cast<const longlong2*>(X + (int64_t)ci[u] * ld + coff[c]));
        }
      if (e + NB <= cnt) {
#pragma unroll
        for (int c = 0; c < MAXCPL; ++c)
          if (mask & (1u << c)) {
#pragma unroll
            for (int u = 0; u < NB; ++u) {
              acc[c][0] += x[u][c].x;
              acc[c][1] += x[u][c].y;
            }
          }
      } else {
#pragma unroll
        for (int c = 0; c < MAXCPL; ++c)
          if (mask & (1u << c)) {
#pragma unroll
            for (int u = 0; u < NB; ++u)
              if (e + u < cnt) {
                acc[c][0] += x[u][c].x;
                acc[c][1] += x[u][c].y;
              }
          }
      }
    }
  }
}
// deg u - S 2^E: the two 32-bit halves of S as exact doubles, every factor made
// from the exponent's bits
__device__ __forceinline__ double lz_fix_row(long long S, double deg, double u, int E) {
  // 2^52 + 2^31 + high half, 2^52 + low half
  const double dh = __hiloint2double(0x43300000, (int)((unsigned long long)S >> 32) ^ 0x80000000);
  const double dl = __hiloint2double(0x43300000, (int)S);
  const int x = (E + 1023) << 20;  // (high word of 2^E)
  // both fma are exact: 2^(E+32) (2^52 + 2^31) = 2^(E+84) (1 + 2^-21)
  const double h = fma(__hiloint2double((x + (32 << 20)) | 0x80000000, 0), dh,
                       __hiloint2double(x + (84 << 20), 0x80000000));
  const double l = fma(__hiloint2double(x | 0x80000000, 0), dl, __hiloint2double(x + (52 << 20), 0));
  return fma(deg, u, h) + l;
}

// (SQ: w^T w as a third sum, from which the fixed-point unit of u_{k+1} is made;
// NBX: entries in flight, 0: the most the instance's registers hold)
template <typename T, int MAXCPL, bool VF, bool FX = false, bool SQ = FX, int NBX = 0>
__device__ __forceinline__ void lz_dots_body(const LzArgs<T>& a, const Blk& blk) {
  static_assert(!FX || (VF && sizeof(T) == 8), "fixed-point sums: unit weights, double");
  using C = c2<T>;
  constexpr int NC = sizeof(T) == 4 ? 2 : 1, V = LZV<T>, NS = SQ ? 3 : 2;
  if (__ldcg(&a.ctl->done)) return;
  const RowMap mp = row_map(a.lanes, a.cpl, blk);
  const unsigned gmask = group_mask(mp.G);
  const int qbase = blk.y * mp.G * mp.cpl + mp.lg;
  const int k = __ldcg(&a.dyn->k);
  const T* __restrict__ U = (const T*)__ldcg((const unsigned long long*)&a.dyn->du);
  int coff[MAXCPL];
  unsigned mask = 0;
#pragma unroll
  for (int c = 0; c < MAXCPL; ++c) {
    const int q = qbase + c * mp.G;
    coff[c] = q * V;
    if (c < mp.cpl && q < a.nq && __ldcg(a.qact + q)) mask |= 1u << c;
  }
  T du[MAXCPL][V], dw[MAXCPL][V], dq[MAXCPL][V];
#pragma unroll
  for (int c = 0; c < MAXCPL; ++c)
#pragma unroll
    for (int v = 0; v < V; ++v) du[c][v] = dw[c][v] = dq[c][v] = (T)0;
  if (__any_sync(0xffffffffu, mask != 0)) {
    const int32_t* __restrict__ rowptr = VF ? a.lrowptr : a.rowptr;
    for (int64_t row = mp.gid; row < a.n; row += mp.gstride) {
      const int k0 = __ldg(rowptr + row), k1 = __ldg(rowptr + row + 1);
      C acc[MAXCPL][NC];
#pragma unroll
      for (int c = 0; c < MAXCPL; ++c)
#pragma unroll
        for (int j = 0; j < NC; ++j) acc[c][j] = mk<T>((T)0, (T)0);
      // narrow instances have the registers to keep more entries in flight
      constexpr int NB = NBX ? NBX : MAXCPL == 1 ? 8 : MAXCPL == 2 ? 4 : 2;
      long long fx[MAXCPL][2];
      if constexpr (FX) {
#pragma unroll
        for (int c = 0; c < MAXCPL; ++c) fx[c][0] = fx[c][1] = 0;
        gather_row_fix<MAXCPL, NB>(a.lcolidx, k0, k1, (int)row, mp.lg, mp.G, gmask, a.qu, a.ld, coff,
                                   mask, fx);
      } else if constexpr (VF)
        gather_row_vf<T, NC, MAXCPL, NB>(a.lcolidx, k0, k1, (int)row, mp.lg, mp.G, gmask, U, a.ld,
                                         coff, mask, acc);
      else
        gather_row<T, NC, MAXCPL, NB>(a.colidx, a.val, k0, k1, (int)row, mp.lg, mp.G, gmask, U,
                                      a.ld, coff, mask, acc);
      const T deg = (T)(k1 - k0);
#pragma unroll
      for (int c = 0; c < MAXCPL; ++c)
        if (mask & (1u << c)) {
          C uv[NC], wv[NC];
          ld_chunk<NC>(U + row * a.ld + coff[c], uv);
          if constexpr (FX) {
            // (loaded per row: the registers of the gathers are worth more)
            int E0, E1;
            asm volatile("ld.global.v2.s32 {%0, %1}, [%2];" : "=r"(E0), "=r"(E1) : "l"(a.qe + coff[c]));
            wv[0] = mk<T>(lz_fix_row(fx[c][0], deg, uv[0].x, E0), lz_fix_row(fx[c][1], deg, uv[0].y, E1));
          }
#pragma unroll
          for (int j = 0; j < NC; ++j) {
            // values-free: L u = deg u - (sum over neighbours)
            if constexpr (!FX) wv[j] = VF ? mk<T>(fma(deg, uv[j].x, -acc[c][j].x), fma(deg, uv[j].y, -acc[c][j].y))
                       : acc[c][j];
            du[c][2 * j] = fma(uv[j].x, uv[j].x, du[c][2 * j]);
            du[c][2 * j + 1] = fma(uv[j].y, uv[j].y, du[c][2 * j + 1]);
            dw[c][2 * j] = fma(uv[j].x, wv[j].x, dw[c][2 * j]);
            dw[c][2 * j + 1] = fma(uv[j].y, wv[j].y, dw[c][2 * j + 1]);
            if constexpr (SQ) {
              dq[c][2 * j] = fma(wv[j].x, wv[j].x, dq[c][2 * j]);
              dq[c][2 * j + 1] = fma(wv[j].y, wv[j].y, dq[c][2 * j + 1]);
            }
          }
          st_chunk<NC>(a.w + row * a.ld + coff[c], wv);
        }
    }
  }
  // groups of a warp by shuffles, warps in shared memory in order, CTAs by
  // global atomics
  extern __shared__ double sred[];  // [WARPS][G * MAXCPL * V * NS]
  const int nred = mp.G * MAXCPL * V * NS;
#pragma unroll
  for (int c = 0; c < MAXCPL; ++c)
#pragma unroll
    for (int v = 0; v < V; ++v) {
      double x = (double)du[c][v], y = (double)dw[c][v], z = (double)dq[c][v];
      for (int o = mp.G; o < 32; o <<= 1) {
        x += __shfl_xor_sync(0xffffffffu, x, o);
        y += __shfl_xor_sync(0xffffffffu, y, o);
        if constexpr (SQ) z += __shfl_xor_sync(0xffffffffu, z, o);
      }
      if ((threadIdx.x & 31) < mp.G) {
        double* o = sred + (threadIdx.x >> 5) * nred + ((mp.lg * MAXCPL + c) * V + v) * NS;
        o[0] = x;
        o[1] = y;
        if constexpr (SQ) o[2] = z;
      }
    }
  __syncthreads();
  for (int t = threadIdx.x; t < nred; t += blockDim.x) {
    const int c = (t / (NS * V)) % MAXCPL, lg = t / (NS * V * MAXCPL);
    const int q = blk.y * mp.G * mp.cpl + lg + c * mp.G;
    if (c < mp.cpl && q < a.nq) {
      double x = 0.0;
#pragma unroll
      for (int w = 0; w < WARPS; ++w) x += sred[w * nred + t];
      if (x != 0.0) atomicAdd(&a.acc[NS * (q * V + (t / NS) % V) + t % NS], x);
    }
    __threadfence();
  }
  __syncthreads();
  __shared__ int s_last;
  if (threadIdx.x == 0) s_last = atomicAdd(&a.ctl->ticket, 1u) == (unsigned)(blk.gx * blk.gy) - 1;
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  for (int t = threadIdx.x; t < NS * a.ld; t += blockDim.x) {
    sred[t] = __ldcg(a.acc + t);
    a.acc[t] = 0.0;
  }
  __syncthreads();
  if (!a.dry) lz_column_scalars<T, NS>(a, k, 0, a.ld, sred);  // (dry: a timing run)
  // (the last thread, which has no column: two latency chains side by side)
  if (threadIdx.x == blockDim.x - 1) {
    if (!a.dry) lz_advance<T>(a, k);
    a.ctl->ticket = 0;
    __threadfence();
  }
}
template <typename T>
__host__ __device__ inline size_t lz_dots_smem(int lanes, int maxcpl, int ld, int ns = 2) {
  const size_t red = (size_t)WARPS * lanes * maxcpl * LZV<T> * ns * sizeof(double);
  const size_t sc = (size_t)ld * ns * sizeof(double);
  return red > sc ? red : sc;
}

// ---------------------------------------------------------------------------
// update: u_{k+1} = s (w - alpha u_k - g u_{k-1}), rows [r0, r1) from the top
// (the product wrote its last rows of w and read its last rows of u most
// recently, so a downward walk finds them in L2). A thread keeps one chunk of
// columns, its coefficients in registers. Bound by HBM: 4 real values per row
// and column.
// ---------------------------------------------------------------------------
// FX: u_{k+1} also as rint(u 2^-E) into the fixed-point copy.
template <typename T, bool FX = false>
__device__ __forceinline__ void lz_update_rows(const LzArgs<T>& a, int64_t r0, int64_t r1) {
  using Q = typename LzVec<T>::t;
  constexpr int V = LZV<T>, UN = 4;
  const int nq = a.nq, per = THREADS / nq;
  const int q = threadIdx.x % nq, rs = threadIdx.x / nq;
  if (rs >= per || !__ldcg(a.qact + q)) return;
  T al[V], g[V], s[V];
  int E[V];
#pragma unroll
  for (int v = 0; v < V; ++v) {
    if constexpr (FX) E[v] = a.qe[q * V + v];
    const LzCoef<T> c = a.cf[q * V + v];
    al[v] = -c.alpha;
    g[v] = -c.g;
    s[v] = c.s;
  }
  const T* U = (const T*)__ldcg((const unsigned long long*)&a.dyn->uu) + q * V;
  const T* B = (const T*)__ldcg((const unsigned long long*)&a.dyn->up);
  T* N = (T*)__ldcg((const unsigned long long*)&a.dyn->un) + q * V;
  const bool first = B == nullptr;  // no u_{k-1} yet
  B += q * V;
  const T* W = a.w + q * V;
  for (int64_t r = r1 - 1 - rs; r >= r0; r -= (int64_t)UN * per) {
    Q u[UN], b[UN], w[UN];
#pragma unroll
    for (int x = 0; x < UN; ++x) {
      const int64_t rr = r - (int64_t)x * per;
      if (rr >= r0) {
        const int64_t o = rr * a.ld;
        w[x] = __ldcg(reinterpret_cast<const Q*>(W + o));
        u[x] = __ldcg(reinterpret_cast<const Q*>(U + o));
        if (!first) b[x] = __ldcs(reinterpret_cast<const Q*>(B + o));
      }
    }
#pragma unroll
    for (int x = 0; x < UN; ++x) {
      const int64_t rr = r - (int64_t)x * per;
      if (rr >= r0) {
        T uv[V], bv[V], wv[V];
        lz_get(u[x], uv);
        lz_get(w[x], wv);
        if (!first) lz_get(b[x], bv);
#pragma unroll
        for (int v = 0; v < V; ++v) {
          T y = fma(al[v], uv[v], wv[v]);
          if (!first) y = fma(g[v], bv[v], y);
          wv[v] = s[v] * y;
        }
        *reinterpret_cast<Q*>(N + rr * a.ld) = lz_put(wv);
        if constexpr (FX)
          *reinterpret_cast<longlong2*>(a.qu + rr * a.ld + q * V) =
              make_longlong2(lz_fix(wv[0], E[0]), lz_fix(wv[1], E[1]));
      }
    }
  }
}

// ---------------------------------------------------------------------------
// the chunk of steps [k0, k1) collapsed, one warp per column (lane j: node j):
// c_k into cc[(k - k0) ld + column] and, with `dirs`, b_jk into
// bb[((k - k0) 2 nc + 2 j (+ 1)) ld + column] and (a_j, g_j) into
// hd[(4 j + .) ld + column]. A latency chain over the steps (two dependent
// FP64 products each) that a whole solve pays once.
// ---------------------------------------------------------------------------
template <typename T>
__device__ __forceinline__ void lz_comp_col(const LzArgs<T>& a, const LzRing& ring, int cap, int c,
                                            int k0, int k1, bool dirs, double (*tile)[17]) {
  const int lane = threadIdx.x & 31, nc = a.nc, j = lane < nc ? lane : 0;
  const int64_t sys = (int64_t)c * nc + j;
  const int kc = min(k1, a.col[c].kstop), ks = a.sh[sys].kstop;
  const bool on = lane < nc, goes = ks >= k1, from = on && k0 > 0 && ks > k0;
  double2 ev = make_double2(0.0, 0.0), t = ev, b = make_double2(goes ? 1.0 : 0.0, 0.0);
  for (int kt = (k1 - k0 - 1) / 32 * 32; kt >= 0; kt -= 32) {  // tiles of 32 steps, backwards
    const int top = min(k1 - k0, kt + 32);
    for (int x0 = top - 1; x0 >= kt; x0 -= 4) {
      double2 tt[4], cw[4];
#pragma unroll
      for (int y = 0; y < 4; ++y) {
        const int k = k0 + x0 - y;
        tt[y] = cw[y] = make_double2(0.0, 0.0);
        if (x0 - y >= kt && k < kc) {
          const double2* th = lz_th(a, lz_slot(a, ring, cap, k));
          tt[y] = th[2 * sys];
          cw[y] = th[2 * sys + 1];
        }
      }
#pragma unroll
      for (int y = 0; y < 4; ++y) {
        const int x = x0 - y;
        if (x < kt) break;
        ev = make_double2(cw[y].x + (t.x * ev.x - t.y * ev.y), cw[y].y + (t.x * ev.y + t.y * ev.x));
        if (on) {
          tile[x - kt][j] = ev.x;
          if (dirs) {
            T* o = a.bb + ((int64_t)x * 2 * nc + 2 * j) * a.ld + c;
            o[0] = (T)b.x;
            o[a.ld] = (T)b.y;
          }
        }
        t = tt[y];
        b = make_double2(t.x * b.x - t.y * b.y, t.x * b.y + t.y * b.x);
      }
    }
    __syncwarp();
    if (kt + lane < top) {
      double s = 0.0;
      for (int i = 0; i < nc; ++i) s += tile[lane][i];
      a.cc[(int64_t)(kt + lane) * a.ld + c] = (T)s;
    }
    __syncwarp();
  }
  if (on) {
    // b = a_j; g_j = t_k0 e_k0
    T* o = a.hd + (int64_t)(4 * j) * a.ld + c;
    o[0] = from ? (T)b.x : (T)0;
    o[a.ld] = from ? (T)b.y : (T)0;
    o[2 * a.ld] = from ? (T)(t.x * ev.x - t.y * ev.y) : (T)0;
    o[3 * a.ld] = from ? (T)(t.x * ev.y + t.y * ev.x) : (T)0;
    a.pflag[sys] = (from ? 1 : 0) | (goes ? 2 : 0);
  }
}

// ---------------------------------------------------------------------------
// D += sum_k c_k u_k over the steps [k0, k1), rows [r0, r1): the pass that ends
// a solve whose steps all fit the ring. A thread takes RPT rows of one chunk of
// columns, UB slots' loads in flight together; the coefficients come through
// L1 (one 16-byte read per RPT rows). Bound by HBM: each u read once. Slots past
// a column's stop are read with a coefficient of 0 while its neighbours in the
// chunk go on; lz_column_scalars keeps them finite.
// ---------------------------------------------------------------------------
template <typename T>
__device__ __forceinline__ void lz_sum_rows(const LzArgs<T>& a, const LzRing& ring, int cap, int k0,
                                            int k1, int64_t r0, int64_t r1) {
  using Q = typename LzVec<T>::t;
  constexpr int V = LZV<T>, RPT = 4, UB = 4;
  const int nq = a.nq, per = THREADS / nq;
  const int q = threadIdx.x % nq, rs = threadIdx.x / nq;
  if (rs >= per) return;
  int kq = k0;  // the chunk of columns has coefficients below kq
#pragma unroll
  for (int v = 0; v < V; ++v) kq = max(kq, min(k1, a.col[q * V + v].kstop));
  for (int64_t r = r0 + rs; r < r1; r += (int64_t)RPT * per) {
    int64_t o[RPT];
    T d[RPT][V];
#pragma unroll
    for (int x = 0; x < RPT; ++x) {
      const int64_t rr = r + (int64_t)x * per;
      o[x] = (rr < r1 ? rr : r) * a.ld + q * V;  // (a row past the end repeats the first)
      lz_get(*reinterpret_cast<const Q*>(a.dacc + o[x]), d[x]);
    }
    for (int k = k0; k < kq; k += UB) {
      Q uq[UB][RPT], cq[UB];
#pragma unroll
      for (int y = 0; y < UB; ++y)
        if (k + y < kq) {
          const T* U = (const T*)lz_slot(a, ring, cap, k + y);
          cq[y] = __ldg(reinterpret_cast<const Q*>(a.cc + (int64_t)(k + y - k0) * a.ld + q * V));
#pragma unroll
          for (int x = 0; x < RPT; ++x) uq[y][x] = __ldcs(reinterpret_cast<const Q*>(U + o[x]));
        }
#pragma unroll
      for (int y = 0; y < UB; ++y)
        if (k + y < kq) {
          T c[V];
          lz_get(cq[y], c);
#pragma unroll
          for (int x = 0; x < RPT; ++x) {
            T uv[V];
            lz_get(uq[y][x], uv);
#pragma unroll
            for (int v = 0; v < V; ++v) d[x][v] = fma(c[v], uv[v], d[x][v]);
          }
        }
    }
#pragma unroll
    for (int x = 0; x < RPT; ++x)
      if (r + (int64_t)x * per < r1) *reinterpret_cast<Q*>(a.dacc + o[x]) = lz_put(d[x]);
  }
}

// ---------------------------------------------------------------------------
// a chunk that directions p_j enter or leave: D and up to JB directions from
// node j0 over the steps [k0, k1), rows [r0, r1). A thread takes RPT rows of
// one chunk of columns, so that the 2 JB + 1 coefficients of a step (through
// L1) serve RPT rows. Bound by HBM in float (u once, 4 N_c values of the
// directions per chunk), by the FP64 pipe in double.
// ---------------------------------------------------------------------------
template <typename T, int JB, int RPT>
__device__ __forceinline__ void lz_apply_rows(const LzArgs<T>& a, const LzRing& ring, int cap,
                                              int j0, int k0, int k1, int64_t r0, int64_t r1) {
  using Q = typename LzVec<T>::t;
  constexpr int V = LZV<T>, UB = 2;
  const int nq = a.nq, nc = a.nc, per = THREADS / nq;
  const int q = threadIdx.x % nq, rs = threadIdx.x / nq;
  if (rs >= per) return;
  int kq = k0, fl = 0;
#pragma unroll
  for (int v = 0; v < V; ++v) {
    kq = max(kq, min(k1, a.col[q * V + v].kstop));
#pragma unroll
    for (int j = 0; j < JB; ++j)
      if (j0 + j < nc) fl |= a.pflag[(int64_t)(q * V + v) * nc + j0 + j] << (2 * j);
  }
  if (kq == k0) return;
  const int64_t plane = a.n * (int64_t)a.ld;
  for (int64_t r = r0 + rs; r < r1; r += (int64_t)RPT * per) {
    int64_t o[RPT];
    T d[RPT][V], pr[RPT][JB][V], pi[RPT][JB][V];
#pragma unroll
    for (int x = 0; x < RPT; ++x) {
      const int64_t rr = r + (int64_t)x * per;
      o[x] = (rr < r1 ? rr : r) * a.ld + q * V;
      lz_get(*reinterpret_cast<const Q*>(a.dacc + o[x]), d[x]);
    }
#pragma unroll
    for (int j = 0; j < JB; ++j) {
#pragma unroll
      for (int x = 0; x < RPT; ++x)
#pragma unroll
        for (int v = 0; v < V; ++v) pr[x][j][v] = pi[x][j][v] = (T)0;
      if (fl >> (2 * j) & 1) {
        T h[4][V];
#pragma unroll
        for (int y = 0; y < 4; ++y)
          lz_get(__ldg(reinterpret_cast<const Q*>(a.hd + (int64_t)(4 * (j0 + j) + y) * a.ld + q * V)), h[y]);
#pragma unroll
        for (int x = 0; x < RPT; ++x) {
          T re[V], im[V];
          const T* P = a.p + (int64_t)(2 * (j0 + j)) * plane + o[x];
          lz_get(__ldcs(reinterpret_cast<const Q*>(P)), re);
          lz_get(__ldcs(reinterpret_cast<const Q*>(P + plane)), im);
#pragma unroll
          for (int v = 0; v < V; ++v) {
            d[x][v] = fma(h[2][v], re[v], fma(-h[3][v], im[v], d[x][v]));
            pr[x][j][v] = fma(h[0][v], re[v], -h[1][v] * im[v]);
            pi[x][j][v] = fma(h[0][v], im[v], h[1][v] * re[v]);
          }
        }
      }
    }
    for (int k = k0; k < kq; k += UB) {
      Q uq[UB][RPT];
#pragma unroll
      for (int y = 0; y < UB; ++y)
        if (k + y < kq) {
          const T* U = (const T*)lz_slot(a, ring, cap, k + y);
#pragma unroll
          for (int x = 0; x < RPT; ++x) uq[y][x] = __ldcs(reinterpret_cast<const Q*>(U + o[x]));
        }
#pragma unroll
      for (int y = 0; y < UB; ++y)
        if (k + y < kq) {
          T uv[RPT][V];
#pragma unroll
          for (int x = 0; x < RPT; ++x) lz_get(uq[y][x], uv[x]);
          if (j0 == 0) {
            T c[V];
            lz_get(__ldg(reinterpret_cast<const Q*>(a.cc + (int64_t)(k + y - k0) * a.ld + q * V)), c);
#pragma unroll
            for (int x = 0; x < RPT; ++x)
#pragma unroll
              for (int v = 0; v < V; ++v) d[x][v] = fma(c[v], uv[x][v], d[x][v]);
          }
          const T* bk = a.bb + (int64_t)(k + y - k0) * 2 * nc * a.ld + q * V;
#pragma unroll
          for (int j = 0; j < JB; ++j)
            if (fl >> (2 * j) & 2) {
              T br[V], bi[V];
              lz_get(__ldg(reinterpret_cast<const Q*>(bk + (int64_t)(2 * (j0 + j)) * a.ld)), br);
              lz_get(__ldg(reinterpret_cast<const Q*>(bk + (int64_t)(2 * (j0 + j) + 1) * a.ld)), bi);
#pragma unroll
              for (int x = 0; x < RPT; ++x)
#pragma unroll
                for (int v = 0; v < V; ++v) {
                  pr[x][j][v] = fma(br[v], uv[x][v], pr[x][j][v]);
                  pi[x][j][v] = fma(bi[v], uv[x][v], pi[x][j][v]);
                }
            }
        }
    }
#pragma unroll
    for (int x = 0; x < RPT; ++x) {
      if (r + (int64_t)x * per >= r1) continue;
      *reinterpret_cast<Q*>(a.dacc + o[x]) = lz_put(d[x]);
#pragma unroll
      for (int j = 0; j < JB; ++j)
        if (fl >> (2 * j) & 2) {
          T* P = a.p + (int64_t)(2 * (j0 + j)) * plane + o[x];
          *reinterpret_cast<Q*>(P) = lz_put(pr[x][j]);
          *reinterpret_cast<Q*>(P + plane) = lz_put(pi[x][j]);
        }
    }
  }
}

}  // namespace rafeast
