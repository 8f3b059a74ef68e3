// Order-independent sums of doubles in integer arithmetic, for the latency-bound
// reductions of resident.cu.  GB300 issues one FP64 instruction of a warp in
// 64 cycles per scheduler, so a shuffle tree of FP64 adds over a CTA and then
// over the grid cost 3 to 5 us; here every value becomes a 57-bit integer on
// the scale of the largest one, warps add with redux.sync, and only the final
// total is rounded to a double (to nearest).  Values are truncated at 2^-57
// of the largest of their warp (FP64 addition rounds at 2^-53 of the partial
// sum), and the result does not depend on the order of the additions.
#pragma once
#include <stdint.h>

namespace sem {

__host__ __device__ inline int min_int(int a, int b) { return a < b ? a : b; }

// m 2^(e - 1079), e the biased FP64 exponent of the scale (a sum's may exceed
// 0x7FE: its value need not); e >= kFxInf: not finite
struct FxVal {
  long long m;
  int e;
};
// the exponents of values that are not finite, so that the largest of a sum's tells
// what it is: +Inf, or NaN (-Inf counts as NaN: no sum here survives either)
constexpr int kFxInf = 0xFFF, kFxBad = 0x1000;

// biased exponent of a double (1 for zero and subnormals)
__host__ __device__ inline int fx_exp(unsigned long long bits) {
  const int ex = (int)((bits >> 52) & 0x7FF);
  if (ex == 0x7FF) return bits == 0x7FF0000000000000ull ? kFxInf : kFxBad;
  return ex ? ex : 1;
}

// the double on the scale e >= its own exponent (finite values), truncated
__host__ __device__ inline long long fx_mant(unsigned long long bits, int e) {
  unsigned long long m = bits & 0xFFFFFFFFFFFFFull;
  const int ex = (int)((bits >> 52) & 0x7FF);
  if (ex) m |= 1ull << 52;
  const int sh = e - (ex ? ex : 1);
  m = sh < 58 ? (m << 4) >> sh : 0ull;
  return (bits >> 63) ? -(long long)m : (long long)m;
}

// a float's biased FP32 exponent (1 for zero and subnormals), and the float on the
// scale e >= it, truncated: m 2^(e - 183), the same m as fx_mant's of (double)f
// on the scale e + 896
__host__ __device__ inline int fx_expf(unsigned f) {
  const int ex = (int)((f >> 23) & 0xFFu);
  return ex ? ex : 1;
}
__host__ __device__ inline long long fx_mantf(unsigned f, int e) {
  const int ex = (int)((f >> 23) & 0xFFu), sh = e - (ex ? ex : 1);
  const unsigned long long w = (unsigned long long)((f & 0x7FFFFFu) | (ex ? 0x800000u : 0u)) << 33;
  const long long m = sh < 64 ? (long long)(w >> sh) : 0;
  return (f >> 31) ? -m : m;
}

// (hi 2^32 + lo) 2^(e - 1079) as a double, lo >= 0: rounded to nearest from its
// leading 64 bits
__host__ __device__ inline double fx_round(long long hi, long long lo, int e) {
  hi += lo >> 32;
  unsigned l = (unsigned)lo;
  const bool neg = hi < 0;
  if (neg) {
    l = 0u - l;
    hi = ~hi + (l == 0u ? 1 : 0);
  }
  unsigned long long m = (unsigned long long)hi, bits = neg ? 1ull << 63 : 0ull;
  if (e >= kFxInf) {
    bits = e == kFxInf ? 0x7FF0000000000000ull : 0x7FF8000000000000ull;
  } else if (m | l) {
    // the leading 64 bits, bit 63 set; ex: the biased exponent of bit 63
#ifdef __CUDA_ARCH__
    const int n = m ? __clzll((long long)m) : 32 + __clz((int)l) + 32;
#else
    const int n = m ? __builtin_clzll(m) : 64 + __builtin_clz(l);
#endif
    if (m) m = (m << n) | (n >= 32 ? (unsigned long long)l << (n - 32) : (unsigned long long)(l >> (32 - n)) * (n != 0));
    else m = (unsigned long long)l << (n - 32);
    int ex = e + 95 - n - 56;
    int sh = 11;
    if (ex < 1) {                         // subnormal
      sh = min_int(11 + 1 - ex, 64);
      ex = 0;
    }
    const unsigned long long half = (m >> (sh - 1)) & 1ull;
    m = (sh < 64 ? m >> sh : 0ull) + half;   // up to 2^53: the carry moves the exponent
    if (ex == 0) bits |= m;                  // 2^52: the smallest normal number
    else if (ex >= 0x7FF) bits |= 0x7FF0000000000000ull;
    else bits |= ((unsigned long long)(ex - 1) << 52) + m;
  }
#ifdef __CUDA_ARCH__
  return __longlong_as_double((long long)bits);
#else
  double d;
  __builtin_memcpy(&d, &bits, 8);
  return d;
#endif
}

#ifdef __CUDACC__
// sum over the warp of 64-bit integers, exact; the result in every lane
// (three redux.sync on 27-bit pieces: 32 x 2^27 fits 32 bits)
__device__ __forceinline__ long long fx_warp_add(long long m) {
  const unsigned lo = __reduce_add_sync(0xffffffffu, (unsigned)m & 0x7FFFFFFu);
  const unsigned mi = __reduce_add_sync(0xffffffffu, (unsigned)(m >> 27) & 0x7FFFFFFu);
  const int hi = __reduce_add_sync(0xffffffffu, (int)(m >> 54));
  return ((long long)hi << 54) + ((long long)mi << 27) + (long long)lo;
}

// a b as a double: exact, and of normal factors without the FP64 pipe (two
// conversions and a product are 192 cycles of a scheduler for every warp)
__device__ __forceinline__ double fx_prod(float a, float b) {
  const unsigned ia = __float_as_uint(a), ib = __float_as_uint(b);
  const unsigned ea = (ia >> 23) & 0xFFu, eb = (ib >> 23) & 0xFFu;
  if (ea - 1u < 254u && eb - 1u < 254u) {
    const unsigned long long m = (unsigned long long)((ia & 0x7FFFFFu) | 0x800000u) *
                                 ((ib & 0x7FFFFFu) | 0x800000u);   // 2^46 .. 2^48
    const unsigned top = (unsigned)(m >> 47);
    const unsigned long long bits = ((unsigned long long)((ia ^ ib) >> 31) << 63) |
                                    ((unsigned long long)(ea + eb + 769u + top) << 52) |
                                    ((m << (6u - top)) & 0xFFFFFFFFFFFFFull);
    return __longlong_as_double((long long)bits);
  }
  if (ea < 255u && eb < 255u && (a == 0.0f || b == 0.0f)) return 0.0;
  return (double)a * (double)b;
}

// sum of v over the warp (in every lane): |m| < 2^62
__device__ __forceinline__ FxVal fx_warp_sum(double v) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(v);
  FxVal r;
  r.e = (int)__reduce_max_sync(0xffffffffu, (unsigned)fx_exp(b));
  r.m = r.e >= kFxInf ? 0 : fx_warp_add(fx_mant(b, r.e));
  return r;
}

// the same of compensated FP32 sums s - c (the FP64 pipe takes 64 cycles for every
// conversion)
__device__ __forceinline__ FxVal fx_warp_sum(float s, float c) {
  const unsigned us = __float_as_uint(s), uc = __float_as_uint(c);
  const int e = (int)__reduce_max_sync(0xffffffffu, (unsigned)max(fx_expf(us), fx_expf(uc)));
  if (e == 255) return fx_warp_sum((double)s - (double)c);
  // one bit up: both mantissas are below 2^56
  return FxVal{fx_warp_add(fx_mantf(us, e + 1) - fx_mantf(uc, e + 1)), e + 897};
}

// running sum of FxVals by one lane, on a common scale e fixed beforehand:
// the two halves are added separately, so nothing overflows below 2^31 terms
struct FxAcc {
  long long hi = 0, lo = 0;
  __device__ __forceinline__ void add(FxVal v, int e) {
    const int sh = e - v.e;
    const long long m = sh < 63 ? v.m >> sh : 0;
    hi += m >> 32;
    lo += (long long)(unsigned)m;
  }
};

// Sum of the lanes' accumulators (in every lane), |hi| and lo below 2^50.
__device__ __forceinline__ FxAcc fx_warp_add(const FxAcc& a) {
  FxAcc t;
  const unsigned l0 = __reduce_add_sync(0xffffffffu, (unsigned)a.lo & 0x7FFFFFFu);
  const unsigned l1 = __reduce_add_sync(0xffffffffu, (unsigned)(a.lo >> 27));
  const unsigned h0 = __reduce_add_sync(0xffffffffu, (unsigned)a.hi & 0x7FFFFFFu);
  const int h1 = __reduce_add_sync(0xffffffffu, (int)(a.hi >> 27));
  t.lo = ((long long)l1 << 27) + (long long)l0;
  t.hi = ((long long)h1 << 27) + (long long)h0;
  return t;
}

// Sum of the lanes' FxVals, in every lane
struct FxTot {
  FxAcc acc;
  int e;
};
__device__ __forceinline__ FxTot fx_lane_sum(FxVal f) {
  FxTot t;
  t.e = (int)__reduce_max_sync(0xffffffffu, (unsigned)f.e);
  if (t.e < kFxInf) t.acc.add(f, t.e);
  t.acc = fx_warp_add(t.acc);
  return t;
}
// the sum as one FxVal, sh bits to the right so that it fits
__device__ __forceinline__ longlong2 fx_pack(const FxTot& t, int sh) {
  return make_longlong2((t.acc.hi << (32 - sh)) + (t.acc.lo >> sh),
                        t.e < kFxInf ? t.e + sh : t.e);
}

// sum of v over a CTA of NW warps, in every thread (two barriers; sw: NW entries
// of shared memory)
template <int NW>
__device__ __forceinline__ double fx_block_total(double v, FxVal* sw) {
  const int lane = threadIdx.x & 31;
  const FxVal f = fx_warp_sum(v);
  __syncthreads();
  if (lane == 0) sw[threadIdx.x >> 5] = f;
  __syncthreads();
  const FxTot t = fx_lane_sum(lane < NW ? sw[lane] : FxVal{0, 1});
  return fx_round(t.acc.hi, t.acc.lo, t.e);
}
#endif

}  // namespace sem
