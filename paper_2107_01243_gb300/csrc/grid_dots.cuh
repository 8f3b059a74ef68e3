// Sums over a grid whose CTAs are all resident (a cooperative launch), which is
// also its barrier; the waits are bounded.
#pragma once
#include "sem_internal.cuh"
#include "tma.cuh"
#include "fixsum.cuh"

namespace sem {

// Sums v over the grid.  Warps and the CTA add their values in integer
// arithmetic (fixsum.cuh); warp q (q < NV; modulo the warps) makes the CTA's
// sum of value q, stores it in partials (16 bytes each, NV gridDim.x of them),
// arrives at the grid barrier, waits (bounded) for target arrivals, NV a CTA,
// and adds the partials: every CTA the same way, so all get the same totals.
// Then thread 0 steps the state.  False when the wait ran out.
template <int NV, int NW, class F>
__device__ __forceinline__ bool grid_dots(const double (&v)[NV], FxVal (*sw)[16], longlong2* sp,
                                          double* tot, longlong2* partials, unsigned* bar,
                                          unsigned target, int* err, uint64_t timeout_ns,
                                          int* s_bad, F step) {
  static_assert(NW <= 16, "a slot per warp");
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nb = gridDim.x;
#pragma unroll
  for (int q = 0; q < NV; ++q) {
    const FxVal f = fx_warp_sum(v[q]);
    if (lane == 0) sw[q][warp] = f;
  }
  __syncthreads();
  for (int q = warp; q < NV; q += NW) {
    const FxTot t = fx_lane_sum(lane < NW ? sw[q][lane] : FxVal{0, 1});
    if (lane == 0) {                     // at most 16 x 2^62
      __stcg(partials + q * nb + blockIdx.x, fx_pack(t, 4));
      asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(bar) : "memory");
    }
  }
  for (int q = warp; q < NV; q += NW) {
    if (lane == 0) {
      unsigned seen;
      uint64_t t0 = 0;
      for (uint32_t it = 1;; ++it) {
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(bar) : "memory");
        if (seen >= target) break;
        if ((it & 255u) == 0) {
          if (t0 == 0) t0 = global_timer_ns();
          if (global_timer_ns() - t0 > timeout_ns || it == 0) {
            atomicExch(err, (int)SEM_ERR_TIMEOUT);
            *s_bad = 1;
            break;
          }
        }
      }
    }
    __syncwarp();
    longlong2* mine = sp + q * nb;
    unsigned e = 1u;
#pragma unroll 4
    for (int l = lane; l < nb; l += 32) {
      const longlong2 p = __ldcg(partials + q * nb + l);
      mine[l] = p;
      e = max(e, (unsigned)p.y);
    }
    e = __reduce_max_sync(0xffffffffu, e);
    FxAcc acc;
    if (e < kFxInf)
      for (int l = lane; l < nb; l += 32) acc.add(FxVal{mine[l].x, (int)mine[l].y}, (int)e);
    acc = fx_warp_add(acc);
    if (lane == 0) tot[q] = fx_round(acc.hi, acc.lo, (int)e);
  }
  __syncthreads();
  if (tid == 0) step();
  __syncthreads();
  return *s_bad == 0;
}

// bits of a double: FP64 comparisons cost as much as additions
__device__ __forceinline__ long long dbits(double v) { return __double_as_longlong(v); }
__device__ __forceinline__ bool is_nan(double v) {
  return (dbits(v) & ~(1ll << 63)) > 0x7FF0000000000000ll;
}

}  // namespace sem
