// Staging of row tiles in shared memory, shared by the tiled sparse products
// (kernels_tiled.cu, kernels_lz_tiled.cu): asynchronous 16-byte copies, packed
// float arithmetic and the staged index data of a tile.
#pragma once

#include <cstddef>

#include "common.cuh"
#include "internal.h"

namespace rafeast {

// threads per CTA and the CTAs per SM the kernel is compiled for
#ifndef RF_TILED_TT
#define RF_TILED_TT 256
#endif
constexpr int TT = RF_TILED_TT;
constexpr int TT_MINB = TT == 256 ? 3 : 6;

__device__ __forceinline__ void cp_async16(void* smem, const void* gmem) {
  const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(s), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() {
  asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;\n" ::: "memory");
}

// a 16-byte chunk as two packed float pairs; add.rn.f32x2 / fma.rn.f32x2
// (sm_100 and later) round each lane exactly as two scalar operations would
using u64 = unsigned long long;
struct __align__(16) P4 {
  u64 lo, hi;
};
__device__ __forceinline__ u64 add2(u64 a, u64 b) {
  u64 d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ u64 fma2(u64 a, u64 b, u64 c) {
  u64 d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ P4 p4add(P4 a, P4 b) { return P4{add2(a.lo, b.lo), add2(a.hi, b.hi)}; }
__device__ __forceinline__ P4 p4fma(u64 s2, P4 b, P4 a) {
  return P4{fma2(s2, b.lo, a.lo), fma2(s2, b.hi, a.hi)};
}
__device__ __forceinline__ u64 splat2(float v) {
  const unsigned u = __float_as_uint(v);
  return ((u64)u << 32) | u;
}
__device__ __forceinline__ float2 lo2(u64 v) {
  return make_float2(__uint_as_float((unsigned)v), __uint_as_float((unsigned)(v >> 32)));
}

// the staged index data of one tile (shared memory, one of two buffers)
// (slx first: the 16-byte copies into it need a 16-byte aligned start)
struct __align__(16) TileIdx {
  uint16_t slx[TILE_NNZCAP + 16]; // union positions of the nonzeros, from kbase
  int sidx[TILE_UCAP];            // union rows
  int srp[TILE_TMAX + 1];         // row pointers of the tile's rows
  int r0, nr, nu, us, kbase;
};
static_assert(offsetof(TileIdx, slx) == 0 && sizeof(TileIdx) % 16 == 0,
              "16-byte copies into TileIdx::slx of both buffers must be aligned");
static_assert(sizeof(P4) == 16 && alignof(P4) == 16, "a staged chunk is one aligned 16 bytes");
static_assert((TILE_NNZCAP + 16) % 8 == 0, "slx holds whole 16-byte pieces");

// the copies of one tile (after its indices are in `b` and a barrier): its
// local indices in 16-byte pieces from an aligned start (the array is padded,
// so the last piece stays inside it) and the union's chunks of this column
// block (active pairs only)
template <int CB>
__device__ __forceinline__ void tile_copies(const TileArgs& tl, TileIdx& b, P4* xs,
                                            const float* R, int64_t ldt, int cbk, const int* sact) {
  const int kbase = b.kbase;
  const int npiece = (b.srp[b.nr] - kbase + 7) >> 3;
  for (int c = threadIdx.x; c < npiece; c += TT) cp_async16(b.slx + 8 * c, tl.lidx + kbase + 8 * c);
  for (int idx = threadIdx.x; idx < b.nu * CB; idx += TT) {
    const int jj = idx % CB;
    if (sact[jj])
      cp_async16(xs + idx, R + (int64_t)b.sidx[idx / CB] * ldt + (int64_t)(cbk * CB + jj) * 4);
  }
}

}  // namespace rafeast
