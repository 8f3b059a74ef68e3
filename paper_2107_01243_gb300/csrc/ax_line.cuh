// The line kernels' element body (L-vectors: ax_line.cu; global vectors:
// global.cu and batch_glob.cuh): K consecutive elements a CTA, thread (i, j) of
// an element owning its k-column.
#pragma once
#include "sem_internal.cuh"
#include "ax_tile.cuh"
#include "eo_tile.cuh"

namespace sem {

// Elements per CTA: the most that fit the threads among the counts whose K P^2
// threads fill their warps best.  FP64 at P = 10 takes three (300 of 320 lanes
// instead of 200 of 224: the FP64 pipe is its bound, and pays for idle lanes:
// 818 against 856 us on 8 M points); FP32 there holds 60 G values a thread, and
// two elements fit the registers twice an SM (59 against 64 us).
constexpr int line_elems(int P, bool f64, int threads = 256) {
  const int P2 = P * P, most = f64 && P == 10 ? 320 : threads;
  int best = 1;
  for (int k = 1; k * P2 <= most; ++k) {
    const int lanes = (k * P2 + 31) / 32 * 32, bl = (best * P2 + 31) / 32 * 32;
    if ((long long)k * bl >= (long long)best * lanes) best = k;
  }
  return best;
}

// threads of the global-vector kernels' CTAs: two elements at N = 7, one at N = 9
// (256 threads, twice the elements: 108 against 100 us and 154 against 147 us on
// 17 M points)
constexpr int kGlobThreads = 128;

template <int P, class T, int MOST = 256>
struct LineCfg {
  static constexpr int P2 = P * P, P3 = P2 * P, K = line_elems(P, sizeof(T) == 8, MOST);
  static constexpr int THREADS = (K * P2 + 31) / 32 * 32;
  static constexpr int RS = P | 1, PL = P * RS, VOL = P * PL;   // rows of odd length
  static constexpr int TS = LineTab<P, T>::EO ? LineTab<P, T>::SIZE : 0;
  static constexpr size_t SMEM = (3 * (size_t)K * VOL + TS) * sizeof(T);
  // CTAs per SM the registers are bounded for (FP64: P = 8 four of 256, P = 10 two of 320 threads;
  // FP32, P = 8: three instead of two, sem_apply on 16.8 M points 120 against 134 us)
  static constexpr int MINB = sizeof(T) == 8 ? (P == 8 ? 4 : 2)
                                             : (P >= 10 ? 512 : P == 8 ? 768 : MOST) / MOST;
};

// y = D x or D^T x for a line in registers
template <int P, class T, bool TRANS, class PUT>
__device__ __forceinline__ void line_dots(const T (&x)[P], const DMat<P, T>& D, const T* tab,
                                          PUT put) {
  if constexpr (LineTab<P, T>::EO) {
    eo_dots<P, T>(x, tab + (TRANS ? EoTab<P>::SIZE : 0), put);
  } else {
#pragma unroll
    for (int i = 0; i < P; ++i) {
      T y = (TRANS ? D.d[i] : D.d[i * P]) * x[0];
#pragma unroll
      for (int l = 1; l < P; ++l) y = fma(TRANS ? D.d[l * P + i] : D.d[i * P + l], x[l], y);
      put(i, y);
    }
  }
}

// This thread's place in its element and the element's shared-memory arrays
template <int P, class T, int MOST = 256>
struct LineThread {
  using C = LineCfg<P, T, MOST>;
  int el, lam, i, j, col, ln_r, ln_s;
  T *tab, *U, *R, *S;
  __device__ __forceinline__ void init(unsigned char* smem) {
    const int tid = threadIdx.x;
    el = tid / C::P2;
    lam = tid - el * C::P2;
    i = lam % P;
    j = lam / P;
    col = j * C::RS + i;                 // (i, j, 0)
    ln_r = lam * C::RS;                  // r-line (j, k) = (lam % P, lam / P)
    ln_s = j * C::PL + i;                // s-line (i, k) = (lam % P, lam / P)
    tab = reinterpret_cast<T*>(smem);
    U = tab + C::TS + (el < C::K ? el : 0) * C::VOL;
    R = U + C::K * C::VOL;
    S = R + C::K * C::VOL;
  }
};

// out = (h1 D^T G D + h2 B) u at the k-column: uc the column of u, g, b, h1f the
// element's G, B and h1 at this thread's (i, j, 0) (h1f NULL without; FP32: FIELD tells).  All
// threads of the CTA call it (act: the thread has an element); U is free once
// the second barrier is behind.  PREG: components of G an FP32 thread fetches
// before the forward lines (the rest where they are used).
// FIELD: h1f is given; an FP32 thread fetches its column with G (where it is used its
// latency shows: FP32 sem_ax / sem_apply, us, late / with G / the kernels this one
// took the place of: N = 5, 13,824 elements 26 / 19.6 / 23 and 40 / 31 / 37, N = 7, 4,096
// 22.5 / 15.9 / 16.3 and 28 / 22.5 / 27, N = 9, 5,832 82 / 44 / 45 and 94 / 59 / 64).
template <int PREG = 6, bool FIELD = false, int P, class T, int MOST>
__device__ __forceinline__ void line_element(const LineThread<P, T, MOST>& t, bool act,
                                             const DMat<P, T>& D, const T (&uc)[P], const T* g,
                                             const T* b, const T* h1f, T h1, T h2, T (&out)[P]) {
  using C = LineCfg<P, T, MOST>;
  constexpr int P2 = C::P2, P3 = C::P3, RS = C::RS, PL = C::PL;
  constexpr bool PRE = sizeof(T) == 4;       // prefetches to registers
  // B comes with G where the backward lines are too short to hide its latency and no
  // other CTA hides it (N = 3, cold caches: sem_apply_global on 216 elements 9.7
  // against 11.0 us, sem_apply 11.0 against 11.6); on large grids that costs 1 to 2%
  const bool early_b = PRE && P <= 4 && gridDim.x < 1024;
  T gr[PRE ? P : 1][6], bk[PRE ? P : 1], hk[PRE && FIELD ? P : 1];
  auto fetch_b = [&] {
#pragma unroll
    for (int k = 0; k < P; ++k) bk[PRE ? k : 0] = __ldcs(b + k * P2);
  };
  if (act) {
    if (early_b && h2 != T(0)) fetch_b();
    if constexpr (PRE) {
#pragma unroll
      for (int k = 0; k < P; ++k)
#pragma unroll
        for (int c = 0; c < PREG; ++c) gr[k][c] = __ldcs(g + c * P3 + k * P2);
    }
    if constexpr (PRE && FIELD) {
#pragma unroll
      for (int k = 0; k < P; ++k) hk[k] = __ldcs(h1f + k * P2);
    }
#pragma unroll
    for (int k = 0; k < P; ++k) t.U[k * PL + t.col] = uc[k];
  }
  __syncthreads();
  if (act) {
    T x[P];
#pragma unroll
    for (int l = 0; l < P; ++l) x[l] = t.U[t.ln_r + l];
    line_dots<P, T, false>(x, D, t.tab, [&](int a, T y) { t.R[t.ln_r + a] = y; });
#pragma unroll
    for (int l = 0; l < P; ++l) x[l] = t.U[t.ln_s + l * RS];
    line_dots<P, T, false>(x, D, t.tab, [&](int a, T y) { t.S[t.ln_s + a * RS] = y; });
  }
  __syncthreads();
  T wt[P];
  if (act) {
    T ut[P];
    line_dots<P, T, false>(uc, D, t.tab, [&](int a, T y) { ut[a] = y; });
    const bool field = PRE ? FIELD : h1f != nullptr;
    const bool scale = field || h1 != T(1);
#pragma unroll
    for (int k = 0; k < P; ++k) {
      const T ur = t.R[k * PL + t.col], us = t.S[k * PL + t.col];
      T gq[6];
#pragma unroll
      for (int c = 0; c < 6; ++c)
        gq[c] = PRE && c < PREG ? gr[PRE ? k : 0][c] : __ldcs(g + c * P3 + k * P2);
      const T g11 = gq[0], g22 = gq[1], g33 = gq[2], g12 = gq[3], g13 = gq[4], g23 = gq[5];
      T wr = fma(g13, ut[k], fma(g12, us, g11 * ur));
      T ws = fma(g23, ut[k], fma(g22, us, g12 * ur));
      T wk = fma(g33, ut[k], fma(g23, us, g13 * ur));
      if (scale) {
        const T c = !field ? h1 : PRE ? hk[PRE && FIELD ? k : 0] : __ldcs(h1f + k * P2);
        wr *= c;
        ws *= c;
        wk *= c;
      }
      t.R[k * PL + t.col] = wr;
      t.S[k * PL + t.col] = ws;
      wt[k] = wk;
    }
  }
  if (PRE && !early_b && act && h2 != T(0)) fetch_b();   // on its way during the backward lines
  __syncthreads();
  if (act) {
    T x[P];
#pragma unroll
    for (int l = 0; l < P; ++l) x[l] = t.R[t.ln_r + l];
    line_dots<P, T, true>(x, D, t.tab, [&](int a, T y) { t.R[t.ln_r + a] = y; });
#pragma unroll
    for (int l = 0; l < P; ++l) x[l] = t.S[t.ln_s + l * RS];
    line_dots<P, T, true>(x, D, t.tab, [&](int a, T y) { t.S[t.ln_s + a * RS] = y; });
    line_dots<P, T, true>(wt, D, t.tab, [&](int a, T y) { out[a] = y; });
  }
  __syncthreads();
  if (act) {
#pragma unroll
    for (int k = 0; k < P; ++k) out[k] += t.R[k * PL + t.col] + t.S[k * PL + t.col];
    if (h2 != T(0)) {
#pragma unroll
      for (int k = 0; k < P; ++k)
        out[k] = fma(h2 * (PRE ? bk[PRE ? k : 0] : __ldcs(b + k * P2)), uc[k], out[k]);
    }
  }
}

// Whether the line kernel is this precision's element kernel.  FP32: always
// (8 M points, us, against the kernel it took the place of: N = 2 58 / 79, N = 4
// 50 / 76, N = 6 49 / 99, N = 8 52 / 91; against the bulk-copy kernel, which
// stays for large meshes at N = 7 and 9 and for tuned handles: N = 1 58 / 209,
// N = 3 46 / 52, N = 5 45 / 56, N = 7 42 / 42, N = 9 59 / 61; on 27 to 1,000
// elements sem_apply takes 0.40 to 0.85 of the former kernels' time).  IEEE FP64:
// the orders of the even-odd split from kLineElems64 elements (8 M points, against
// the one-element kernel: N = 7 681 / 783, N = 9 818 / 923; sem_apply on 1,728
// elements 92 / 98 and 200 / 222, on 1,000 65 / 59 and 152 / 129, on 64 34 / 13 and
// 52 / 23: a CTA's four or three elements are a chain four or three times as long
// on the FP64 pipe).  Elsewhere the column kernel (N = 6, 8,000 elements 298 against
// 329 us with plain lines), nor where a handle insists on the double-float kernel.
constexpr int64_t kLineElems64 = 1536;
template <class T>
inline bool line_ax_supported(const sem_handle* h) {
  return sizeof(T) == 4 || (eo_split(h->P, true) && h->E >= kLineElems64 &&
                            h->f64_kernel != SEM_F64_KERNEL_DOUBLEFLOAT);
}

// w = (h1 A + h2 B) u on L-vectors; fuse: masked points zero, x-pairs inside
// segments of line_elems(P, T) elements summed.  st may be null.
template <class T>
void launch_ax_line(const sem_handle* h, const OpData<T>& op, const T* u, T* w, T h1, T h2,
                    const T* h1f, bool fuse, const CGState* st, cudaStream_t s);

}  // namespace sem
