// Jacobi-PCG iterations of small problems in one launch (arXiv 2107.01243 §2
// end; the recurrences of cg.cu).
//
// What bounds small solves is latency: with one kernel per stage an iteration
// on 4^3 elements (N = 7, FP64) took 38 us in six launches, for about 3 us of
// arithmetic.  Here the whole grid stays on the GPU (a cooperative launch of
// at most the resident CTAs).  An iteration takes two grid barriers:
//   - p = z + beta p; the element operator; the local products (masked, not
//     assembled) go to w, and <p, H p> = sum_L p (H_L p) (p is continuous and
//     zero on Dirichlet points, so the sum over local points is the unique-dof
//     product); barrier, alpha
//   - every point gathers the copies of its w (at most eight, summed pair by
//     pair along x, y, z as sem_apply does), x += alpha p, r -= alpha w,
//     z = dinv r, <r, z> and <r, r>; barrier, beta
// (One barrier would do with the recurrences of Chronopoulos and Gear, which
// form <p, H p> from <z, H z> and s = H p by a recurrence; but they lose digits:
// FP32 inner solves took 5 to 20% more iterations, and the residual that FP64
// solves end at was 1% larger, 5 to 10 times with the double-float operator.)
// x, r and p of an element are only touched by its own CTA's threads; w
// alone crosses CTAs, and is read past L1.  Every CTA adds the CTAs' sums the
// same way and steps its own copy of the CGState.  The barrier's wait is
// bounded: a CTA that gives up records SEM_ERR_TIMEOUT and leaves, and the
// others follow.
//
// Microseconds an iteration, resident against one kernel per stage, on 4^3 / 8^3
// elements: FP64 N = 7 11.6 (35.3) / 24.6 (45.2), N = 6 (IEEE) 16.0 (54.7) /
// 39.2 (57.7), FP32 N = 7 9.7 (20.0 on global vectors) / 15.5 (22.5).  On 4^3, N = 7, FP64 the
// operator takes 2.3 us, each barrier with its sums 2.5 us (0.45 of them an FP64
// division), updates and dots on the FP64 pipe 2 us, the copies' reads 1 us.
// FP64 shuffle trees for the sums (fixsum.cuh says why not) took 3 to 5 us each.
#include <type_traits>

#include "sem_internal.cuh"
#include "tma.cuh"
#include "df_tile.cuh"
#include "ax_tile.cuh"
#include "eo_tile.cuh"
#include "grid_dots.cuh"
#include "cg_state.cuh"

namespace sem {

template <class T>
struct ResArgs {
  T *x, *r, *p, *w;           // L-vectors
  const T* dinv;
  const float* imult;
  const void *G, *B;          // T values, or float pairs (double-float operator)
  const T* h1f;               // per-point h1 or NULL
  const T* tab;               // IEEE operators: LineTab
  const int* esc;             // double-float: exponents of G and B per element
  T h1, h2;
  DFScal df;                  // double-float: h1 and h2
  FuseBox fb;
  FastDiv dnx, dny;
  CGState* st;
  longlong2* partials;        // 2 x 2 gridDim.x values
  unsigned* bar;              // zero at launch
  int* err;
  uint64_t timeout_ns;
  int E, iters;
};

// ------------------------------------------------------------ element operators
// out[m] = (H_L in) at this thread's points q = tid + m NT (NT = 3 P^2: a
// thread's points share i and j); all threads of the CTA call it.

// double-float (FP64-accurate on the FP32 pipes): the phases and the range
// handling of ax_df_kernel
template <int P>
struct OpDF {
  using T = double;
  using L = DFLayout<P>;
  static constexpr int P2 = P * P, P3 = P2 * P, NT = 3 * P2, NTB = (NT + 31) / 32 * 32;
  static constexpr int NQ = (P3 + NT - 1) / NT, NW = NTB / 32;
  static constexpr size_t SMEM = 4 * (size_t)L::VOL * sizeof(float2);
  float2 *U, *R0, *R1, *R2, *my;
  int loff[P], qoff[NQ];
  bool act;
  __device__ __forceinline__ void init(unsigned char* smem, const ResArgs<T>&) {
    U = reinterpret_cast<float2*>(smem);
    R0 = U + L::VOL;
    R1 = R0 + L::VOL;
    R2 = R1 + L::VOL;
    const int tid = threadIdx.x, g = tid / P2, lam = tid % P2, c1 = lam % P, c2 = lam / P;
    act = tid < NT;
    my = g == 0 ? R0 : (g == 1 ? R1 : R2);
#pragma unroll
    for (int l = 0; l < P; ++l)
      loff[l] = g == 0 ? L::at(l, c1, c2) : (g == 1 ? L::at(c1, l, c2) : L::at(c1, c2, l));
#pragma unroll
    for (int m = 0; m < NQ; ++m) {
      const int q = tid + m * NT;
      qoff[m] = act && q < P3 ? L::at(q % P, (q / P) % P, q / P2) : 0;
    }
  }
  __device__ __forceinline__ bool has(int m) const {
    return act && ((m + 1) * NT <= P3 || (int)threadIdx.x + m * NT < P3);
  }
  __device__ __forceinline__ void apply(const ResArgs<T>& a, int e, const double (&in)[NQ],
                                        double (&out)[NQ]) {
    __shared__ unsigned s_key[NW];
    const int tid = threadIdx.x;
    const bool helm = a.df.h2h != 0.0f;
    const float2* g = static_cast<const float2*>(a.G) + (size_t)e * 6 * P3;
    // G is on its way while the forward lines run
    float2 gr[NQ][6];
#pragma unroll
    for (int m = 0; m < NQ; ++m)
#pragma unroll
      for (int c = 0; c < 6; ++c)
        gr[m][c] = has(m) ? __ldg(g + c * P3 + tid + m * NT) : make_float2(0.0f, 0.0f);
    const int sw = __ldg(a.esc + e);
    unsigned key = 0u, lor = 0u;
#pragma unroll
    for (int m = 0; m < NQ; ++m) {
      if (has(m)) {
        const unsigned long long xb = (unsigned long long)__double_as_longlong(in[m]);
        key = max(key, (unsigned)(xb >> 32) & 0x7FFFFFFFu);
        lor |= (unsigned)xb;
        float hi, lo;
        d2df(in[m], hi, lo);
        U[qoff[m]] = make_float2(hi, lo);
      }
    }
    key |= (lor != 0u) ? 1u : 0u;
    const unsigned wkey = __reduce_max_sync(0xffffffffu, key);
    if ((tid & 31) == 0) s_key[tid >> 5] = wkey;
    const bool wbad = wkey != 0u && (wkey - kDfKeyLo) >= (kDfKeyHi - kDfKeyLo);
    int kU = 0;
    bool nanel = false;
    if (__syncthreads_or(wbad)) {
      unsigned km = 0u;
#pragma unroll
      for (int w2 = 0; w2 < NW; ++w2) km = max(km, s_key[w2]);
      if (km >= kDfKeyNonFinite) {
        nanel = true;
      } else if (km < kDfKeyLo || km >= kDfKeyHi) {
        kU = df_key_exp(km);
        const int ka = -kU / 2;
        const double sa = df_pow2d(ka), sb = df_pow2d(-kU - ka);
#pragma unroll
        for (int m = 0; m < NQ; ++m)
          if (has(m)) {
            float hi, lo;
            d2df(in[m] * sa * sb, hi, lo);
            U[qoff[m]] = make_float2(hi, lo);
          }
      }
      __syncthreads();
    }
    if (act) line_task<P, false>(U, my, loff);
    const int a1 = (int)(short)(sw & 0xFFFF) + a.df.t1;
    const int a2 = helm ? (sw >> 16) + a.df.t2 : a1;
    const int unit = max(a1, a2);
    const float c1h = df_scale_down(a.df.h1h, a1 - unit), c1l = df_scale_down(a.df.h1l, a1 - unit);
    const bool scale1 = !(c1h == 1.0f && c1l == 0.0f);
    __syncthreads();
#pragma unroll
    for (int m = 0; m < NQ; ++m) {
      if (!has(m)) break;
      const int at = qoff[m];
      const float2 g11 = gr[m][0], g22 = gr[m][1], g33 = gr[m][2];
      const float2 g12 = gr[m][3], g13 = gr[m][4], g23 = gr[m][5];
      const float2 ur = R0[at], us = R1[at], ut = R2[at];
      float rh, rl, sh, sl, th, tl;
      const float mg = fmaxf(fmaxf(fmaxf(fabsf(g11.x), fabsf(g22.x)),
                                   fmaxf(fabsf(g33.x), fabsf(g12.x))),
                             fmaxf(fabsf(g13.x), fabsf(g23.x)));
      const float mu = fmaxf(fmaxf(fabsf(ur.x), fabsf(us.x)), fabsf(ut.x));
      const float sig = df_pow2_ceil(__fmul_rn(__fmul_rn(mg, 3.0f * (1.0f + 0x1p-18f)), mu));
      dot3_x(g11, g12, g13, ur, us, ut, sig, rh, rl);
      dot3_x(g12, g22, g23, ur, us, ut, sig, sh, sl);
      dot3_x(g13, g23, g33, ur, us, ut, sig, th, tl);
      if (scale1) {
        dfmul(c1h, c1l, rh, rl, rh, rl);
        dfmul(c1h, c1l, sh, sl, sh, sl);
        dfmul(c1h, c1l, th, tl, th, tl);
      }
      R0[at] = make_float2(rh, rl);
      R1[at] = make_float2(sh, sl);
      R2[at] = make_float2(th, tl);
    }
    __syncthreads();
    if (act) line_task_xt<P>(my, my, loff);
    __syncthreads();
    const float c2h = df_scale_down(a.df.h2h, a2 - unit), c2l = df_scale_down(a.df.h2l, a2 - unit);
    const float2* b = static_cast<const float2*>(a.B) + (size_t)e * P3;
#pragma unroll
    for (int m = 0; m < NQ; ++m) {
      out[m] = 0.0;
      if (!has(m)) break;
      const int at = qoff[m];
      const float2 cr = R0[at], cs = R1[at], ct = R2[at];
      float S = cr.x, er = cr.y;
      tadd(cs.x, cs.y, S, er);
      tadd(ct.x, ct.y, S, er);
      if (helm) {
        const float2 bv = __ldg(b + tid + m * NT), uv = U[at];
        float bh, bl;
        dfmul(c2h, c2l, bv.x, bv.y, bh, bl);
        tmac(bh, bl, uv.x, uv.y, S, er);
      }
      double val = (double)S + (double)er;
      if (unit + kU != 0) val = df_ldexp(val, unit + kU);
      if (nanel) val = __longlong_as_double(0x7FF8000000000000ll);
      out[m] = val;
    }
    __syncthreads();                     // the arrays are free for the next element
  }
};

// IEEE arithmetic in T (FP64 or FP32), optional per-point h1
template <int P, class TT>
struct OpIEEE {
  using T = TT;
  using L = EoLayout<P, T>;
  static constexpr int P2 = P * P, P3 = P2 * P, NT = 3 * P2, NTB = (NT + 31) / 32 * 32;
  static constexpr int NQ = (P3 + NT - 1) / NT, TS = LineTab<P, T>::SIZE;
  static constexpr size_t SMEM = (4 * (size_t)L::VOL + TS) * sizeof(T);
  T *U, *R0, *R1, *R2, *my, *tab;
  int loff[P], qoff[NQ];
  bool act;
  __device__ __forceinline__ void init(unsigned char* smem, const ResArgs<T>& a) {
    U = reinterpret_cast<T*>(smem);
    R0 = U + L::VOL;
    R1 = R0 + L::VOL;
    R2 = R1 + L::VOL;
    tab = R2 + L::VOL;
    const int tid = threadIdx.x, g = tid / P2, lam = tid % P2, c1 = lam % P, c2 = lam / P;
    for (int q = tid; q < TS; q += NTB) tab[q] = a.tab[q];
    act = tid < NT;
    my = g == 0 ? R0 : (g == 1 ? R1 : R2);
#pragma unroll
    for (int l = 0; l < P; ++l)
      loff[l] = g == 0 ? L::at(l, c1, c2) : (g == 1 ? L::at(c1, l, c2) : L::at(c1, c2, l));
#pragma unroll
    for (int m = 0; m < NQ; ++m) {
      const int q = tid + m * NT;
      qoff[m] = act && q < P3 ? L::at(q % P, (q / P) % P, q / P2) : 0;
    }
  }
  __device__ __forceinline__ bool has(int m) const {
    return act && ((m + 1) * NT <= P3 || (int)threadIdx.x + m * NT < P3);
  }
  __device__ __forceinline__ void apply(const ResArgs<T>& a, int e, const T (&in)[NQ],
                                        T (&out)[NQ]) {
    const int tid = threadIdx.x;
    const T* g = static_cast<const T*>(a.G) + (size_t)e * 6 * P3;
    T gr[NQ][6];                         // on its way while the forward lines run
#pragma unroll
    for (int m = 0; m < NQ; ++m)
#pragma unroll
      for (int c = 0; c < 6; ++c) gr[m][c] = has(m) ? __ldg(g + c * P3 + tid + m * NT) : T(0);
#pragma unroll
    for (int m = 0; m < NQ; ++m)
      if (has(m)) U[qoff[m]] = in[m];
    __syncthreads();
    if (act) tab_line<P, T, false>(U, my, loff, tab);
    const bool scale = a.h1f || a.h1 != T(1);
    __syncthreads();
#pragma unroll
    for (int m = 0; m < NQ; ++m) {
      if (!has(m)) break;
      const int at = qoff[m];
      const T ur = R0[at], us = R1[at], ut = R2[at];
      T wr = fma(gr[m][4], ut, fma(gr[m][3], us, gr[m][0] * ur));
      T ws = fma(gr[m][5], ut, fma(gr[m][1], us, gr[m][3] * ur));
      T wt = fma(gr[m][2], ut, fma(gr[m][5], us, gr[m][4] * ur));
      if (scale) {
        const T c = a.h1f ? __ldg(a.h1f + (size_t)e * P3 + tid + m * NT) : a.h1;
        wr *= c;
        ws *= c;
        wt *= c;
      }
      R0[at] = wr;
      R1[at] = ws;
      R2[at] = wt;
    }
    __syncthreads();
    if (act) tab_line<P, T, true>(my, my, loff, tab);
    __syncthreads();
    const T* b = static_cast<const T*>(a.B) + (size_t)e * P3;
#pragma unroll
    for (int m = 0; m < NQ; ++m) {
      out[m] = T(0);
      if (!has(m)) break;
      const int at = qoff[m];
      T acc = (R0[at] + R1[at]) + R2[at];
      if (a.h2 != T(0)) acc = fma(a.h2 * __ldg(b + tid + m * NT), in[m], acc);
      out[m] = acc;
    }
    __syncthreads();                     // R is free for the next element
  }
};

// ------------------------------------------------------------ the iteration
// per-thread dot accumulation: FP64 for FP64 vectors, compensated FP32 else
template <class T>
struct ResAcc {
  T s = T(0), c = T(0);
  __device__ __forceinline__ void add(T v) {
    if constexpr (sizeof(T) == 8) {
      s += v;
    } else {
      const float y = __fsub_rn(v, c);
      const float t = __fadd_rn(s, y);
      c = __fsub_rn(__fsub_rn(t, s), y);
      s = t;
    }
  }
  __device__ __forceinline__ void add2(T a, T b) {       // a b
    if constexpr (sizeof(T) == 8) s = fma(a, b, s);
    else add(__fmul_rn(a, b));
  }
  __device__ __forceinline__ double value() const {
    if constexpr (sizeof(T) == 8) return s;
    else return (double)s - (double)c;
  }
};

// 1 / mult (a power of two) in T; to double by moving its exponent bits
template <class T>
__device__ __forceinline__ T res_widen(float f) {
  if constexpr (sizeof(T) == 8)
    return __longlong_as_double((long long)((__float_as_uint(f) >> 23) + 896u) << 52);
  else
    return f;
}

// State transitions with the comparisons on the bits of the doubles (an FP64
// comparison costs as much as an addition); tol2 and <r, r> are not negative.

// the recurrences of cg_state.cuh: after <p, H p>
__device__ __forceinline__ void res_after_pw(CGState* st, double pw) {
  st->pw = pw;
  if (dbits(pw) <= 0 || is_nan(pw)) {
    st->status = SEM_ERR_BREAKDOWN;
    st->done = 1;
  } else {
    st->alpha = st->rz / pw;
  }
}

// and after the update (tot = {<r, z>, <r, r>})
__device__ __forceinline__ void res_after_update(CGState* st, const double* tot) {
  st->iter += 1;
  st->rr = tot[1];
  if (is_nan(tot[0]) || is_nan(tot[1])) {
    st->status = SEM_ERR_BREAKDOWN;
    st->done = 1;
  } else if (dbits(tot[1]) <= dbits(st->tol2)) {
    st->done = 1;
  } else if (st->iter >= st->maxit) {
    st->status = SEM_ERR_NOCONV;
    st->done = 1;
  } else {
    st->beta = tot[0] / st->rz;
    st->rz = tot[0];
  }
}

// RES: every CTA has one element, whose vectors stay in registers.
template <class OP, bool RES>
__global__ void __launch_bounds__(OP::NTB)
pcg_resident_kernel(const __grid_constant__ ResArgs<typename OP::T> a) {
  using T = typename OP::T;
  constexpr int P2 = OP::P2, P3 = OP::P3, NT = OP::NT, NQ = OP::NQ, NW = OP::NTB / 32;
  constexpr int P = P3 / P2, N = P - 1;
  extern __shared__ __align__(16) unsigned char smem[];
  longlong2* sp = reinterpret_cast<longlong2*>(smem + (OP::SMEM + 15) / 16 * 16);
  __shared__ CGState s_st;
  __shared__ FxVal s_w[2][16];
  __shared__ double s_tot[2];
  __shared__ int s_bad;
  const int tid = threadIdx.x;
  if (tid == 0) {
    s_bad = 0;
    s_st = *a.st;
    if (!(s_st.tol2 >= 0.0)) s_st.tol2 = 0.0;
  }
  OP op;
  op.init(smem, a);
  __syncthreads();
  if (s_st.done) return;                 // the same in every CTA
  const int i = tid % P, j = (tid / P) % P, k0 = tid / P2;
  T x[NQ], r[NQ], p[NQ], d[NQ];          // this thread's points of one element
  T z[NQ] = {};                          // dinv r
  float im[NQ];
  ResAcc<T> rz, pw, rr;

  auto load = [&](int e) {
    const size_t base = (size_t)e * P3 + tid;
#pragma unroll
    for (int m = 0; m < NQ; ++m) {
      x[m] = r[m] = p[m] = d[m] = T(0);
      im[m] = 1.0f;
      if (op.has(m)) {
        const size_t q = base + m * NT;
        r[m] = a.r[q];
        d[m] = __ldg(a.dinv + q);
        im[m] = __ldg(a.imult + q);
        x[m] = a.x[q];
        p[m] = a.p[q];
      }
    }
  };
  auto store = [&](int e) {
    const size_t base = (size_t)e * P3 + tid;
#pragma unroll
    for (int m = 0; m < NQ; ++m)
      if (op.has(m)) {
        const size_t q = base + m * NT;
        a.x[q] = x[m];
        a.r[q] = r[m];
        a.p[q] = p[m];
      }
  };
  auto dots = [&](int m) {
    const T rm = r[m] * res_widen<T>(im[m]);
    rr.add2(rm, r[m]);
    rz.add2(rm, z[m]);
  };
  // p = z + beta p and w = H_L p with <p, H p>; w is masked, not assembled
  auto front = [&](int e, T beta, bool first) {
    T hp[NQ];
#pragma unroll
    for (int m = 0; m < NQ; ++m) {
      if (!RES) z[m] = d[m] * r[m];              // else left by the last update
      p[m] = first ? z[m] : fma(beta, p[m], z[m]);
    }
    op.apply(a, e, p, hp);
    const uint32_t re = a.dnx.div((uint32_t)e), ez = a.dny.div(re);
    const int ex = e - (int)re * a.fb.nelx, ey = (int)(re - ez * (uint32_t)a.fb.nely);
    const int f = a.fb.faces;
    const bool mij = ((f & SEM_FACE_XMIN) && ex == 0 && i == 0) ||
                     ((f & SEM_FACE_XMAX) && ex == a.fb.nelx - 1 && i == N) ||
                     ((f & SEM_FACE_YMIN) && ey == 0 && j == 0) ||
                     ((f & SEM_FACE_YMAX) && ey == a.fb.nely - 1 && j == N);
    const bool mz0 = (f & SEM_FACE_ZMIN) && ez == 0;
    const bool mz1 = (f & SEM_FACE_ZMAX) && (int)ez == a.fb.nelz - 1;
#pragma unroll
    for (int m = 0; m < NQ; ++m) {
      if (!op.has(m)) break;
      const int k = k0 + 3 * m;
      const bool masked = mij || (mz0 && k == 0) || (mz1 && k == N);
      a.w[(size_t)e * P3 + tid + m * NT] = masked ? T(0) : hp[m];
    }
#pragma unroll
    for (int m = 0; m < NQ; ++m) {
      if (!op.has(m)) break;
      pw.add2(p[m], hp[m]);
    }
  };
  // gathers the copies of w (summed pair by pair along x, y, z), then
  // x += alpha p, r -= alpha w, z = dinv r and the dots
  auto update = [&](int e, T alpha) {
    const T* w = a.w;
    const size_t base = (size_t)e * P3 + tid;
    const uint32_t re = a.dnx.div((uint32_t)e), ez = a.dny.div(re);
    const int ex = e - (int)re * a.fb.nelx, ey = (int)(re - ez * (uint32_t)a.fb.nely);
    // offsets of a point's copies across its element's faces (0: none)
    const int ox = i == 0 && ex > 0 ? N - P3 : (i == N && ex < a.fb.nelx - 1 ? P3 - N : 0);
    const int sy = a.fb.nelx * P3 - N * P;
    const int oy = j == 0 && ey > 0 ? -sy : (j == N && ey < a.fb.nely - 1 ? sy : 0);
    const int sz = a.fb.nelx * a.fb.nely * P3 - N * P2;
    // the adds of copies no lane of the warp has are skipped (FP64 pipe)
    const bool anyx = __any_sync(0xffffffffu, ox), anyy = __any_sync(0xffffffffu, oy);
    T c[NQ][8];                          // all on their way before the sums
    int oz[NQ];
#pragma unroll
    for (int m = 0; m < NQ; ++m) {
      const int k = k0 + 3 * m;
      oz[m] = k == 0 && ez > 0 ? -sz : (k == N && (int)ez < a.fb.nelz - 1 ? sz : 0);
#pragma unroll
      for (int b = 0; b < 8; ++b) {
        const bool in = op.has(m) && (!(b & 1) || ox) && (!(b & 2) || oy) && (!(b & 4) || oz[m]);
        c[m][b] = in ? __ldcg(w + (long long)(base + m * NT) + ((b & 1) ? ox : 0) +
                              ((b & 2) ? oy : 0) + ((b & 4) ? oz[m] : 0))
                     : T(0);
      }
    }
#pragma unroll
    for (int m = 0; m < NQ; ++m) {
      const bool anyz = __any_sync(0xffffffffu, op.has(m) && oz[m]);
      T v = c[m][0];
      if (anyx) v += c[m][1];
      if (anyy) {
        T v2 = c[m][2];
        if (anyx) v2 += c[m][3];
        v += v2;
      }
      if (anyz) {
        T v4 = c[m][4];
        if (anyx) v4 += c[m][5];
        if (anyy) {
          T v6 = c[m][6];
          if (anyx) v6 += c[m][7];
          v4 += v6;
        }
        v += v4;
      }
      x[m] = fma(alpha, p[m], x[m]);
      r[m] = fma(-alpha, v, r[m]);
      z[m] = d[m] * r[m];
      if (op.has(m)) dots(m);
    }
  };

  const int e0 = blockIdx.x;
  unsigned met = 0;
  // sums over the grid at the n-th set of partials (at most 2 gridDim.x each)
  auto meet = [&](auto nv, const double* v, int n, auto step) {
    constexpr int NV = decltype(nv)::value;
    double vv[NV];
#pragma unroll
    for (int q = 0; q < NV; ++q) vv[q] = v[q];
    met += NV * gridDim.x;
    return grid_dots<NV, NW>(vv, s_w, sp, s_tot, a.partials + n * 2 * gridDim.x, a.bar, met, a.err,
                             a.timeout_ns, &s_bad, step);
  };
  using One = std::integral_constant<int, 1>;
  using Two = std::integral_constant<int, 2>;
  if (RES) load(e0);
  for (int it = 0; it < a.iters; ++it) {
    const T beta = (T)s_st.beta;
    pw = ResAcc<T>();
    for (int e = e0; e < a.E; e += gridDim.x) {
      if (!RES) load(e);
      if (it == 0)                       // a new launch: z of the stored r
#pragma unroll
        for (int m = 0; m < NQ; ++m) z[m] = d[m] * r[m];
      front(e, beta, s_st.iter == 0);
      if (!RES) store(e);
    }
    const double v1[1] = {pw.value()};
    if (!meet(One(), v1, 0, [&] { res_after_pw(&s_st, s_tot[0]); })) break;
    if (s_st.done) break;
    const T alpha = (T)s_st.alpha;
    rz = ResAcc<T>();
    rr = ResAcc<T>();
    for (int e = e0; e < a.E; e += gridDim.x) {
      if (!RES) load(e);
      update(e, alpha);
      if (!RES) store(e);
    }
    const double v2[2] = {rz.value(), rr.value()};
    if (!meet(Two(), v2, 1, [&] { res_after_update(&s_st, s_tot); })) break;
    if (s_st.done) break;
  }
  if (RES) store(e0);
  if (blockIdx.x == 0 && tid == 0) *a.st = s_st;
}

// ------------------------------------------------------------ launch
template <class OP>
constexpr int resident_smem() {
  return (int)((OP::SMEM + 15) / 16 * 16 + 2 * kRedBlocks * sizeof(longlong2));
}

template <class OP, bool RES>
static int resident_occupancy() {
  static const int occ = [] {
    auto kern = pcg_resident_kernel<OP, RES>;
    SEM_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  resident_smem<OP>()));
    int o = 0;
    SEM_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o, kern, OP::NTB,
                                                           resident_smem<OP>()));
    return std::max(1, std::min(o, kRedBlocks / sem_num_sms()));
  }();
  return occ;
}

template <class OP>
static void launch_resident_op(sem_handle* h, ResArgs<typename OP::T>& a, cudaStream_t s) {
  if (!h->res_bar.ptr) h->res_bar.alloc(1);
  if (!h->res_part.ptr) h->res_part.alloc(4 * 2 * kRedBlocks);
  a.bar = h->res_bar.ptr;
  a.partials = reinterpret_cast<longlong2*>(h->res_part.ptr);
  SEM_CUDA(cudaMemsetAsync(a.bar, 0, sizeof(unsigned), s));
  void* args[] = {&a};
  if (a.E <= resident_occupancy<OP, true>() * sem_num_sms()) {
    SEM_CUDA(cudaLaunchCooperativeKernel(pcg_resident_kernel<OP, true>, dim3(a.E), dim3(OP::NTB),
                                         args, resident_smem<OP>(), s));
    return;
  }
  const int most = resident_occupancy<OP, false>() * sem_num_sms();
  const int rounds = (a.E + most - 1) / most;
  const int grid = (a.E + rounds - 1) / rounds;      // every CTA the same share (+- 1)
  SEM_CUDA(cudaLaunchCooperativeKernel(pcg_resident_kernel<OP, false>, dim3(grid), dim3(OP::NTB),
                                       args, resident_smem<OP>(), s));
}

template <class T>
static void resident_common(sem_handle* h, const PcgVecs<T>& v, ResArgs<T>& a, int iters) {
  a.x = v.x; a.r = v.r; a.p = v.p; a.w = v.w;
  a.dinv = v.dinv;
  a.imult = h->imult.ptr;
  a.h1f = v.h1f;
  a.h1 = v.h1;
  a.h2 = v.h2;
  a.fb = FuseBox{h->nelx, h->nely, h->nelz, h->faces};
  a.dnx = FastDiv((uint32_t)h->nelx);
  a.dny = FastDiv((uint32_t)h->nely);
  a.st = v.st;
  a.err = h->dev_err.ptr;
  a.timeout_ns = kWaitTimeoutNs;
  a.E = (int)h->E;
  a.iters = iters;
}

template <class T>
static void launch_resident_ieee(sem_handle* h, const T* D, ResArgs<T>& a, cudaStream_t s) {
  auto go = [&](auto p) {
    constexpr int P = decltype(p)::value;
    a.tab = D + LineTab<P, T>::FROM;
    launch_resident_op<OpIEEE<P, T>>(h, a, s);
  };
  switch (h->P) {
    case 2: go(std::integral_constant<int, 2>()); break;
    case 3: go(std::integral_constant<int, 3>()); break;
    case 4: go(std::integral_constant<int, 4>()); break;
    case 5: go(std::integral_constant<int, 5>()); break;
    case 6: go(std::integral_constant<int, 6>()); break;
    case 7: go(std::integral_constant<int, 7>()); break;
    case 8: go(std::integral_constant<int, 8>()); break;
    case 9: go(std::integral_constant<int, 9>()); break;
    case 10: go(std::integral_constant<int, 10>()); break;
    case 11: go(std::integral_constant<int, 11>()); break;
    default: throw Error(SEM_ERR_ARG, "resident CG: unsupported order");
  }
}

template <>
void launch_resident<double>(sem_handle* h, const PcgVecs<double>& v, int iters, cudaStream_t s) {
  ResArgs<double> a{};
  resident_common(h, v, a, iters);
  if (h->f64_kernel != SEM_F64_KERNEL_NATIVE && df_ax_supported(h, v.p, v.w, v.h1f)) {
    a.G = h->gdf.ptr;
    a.B = h->bdf.ptr;
    a.esc = h->escale.ptr;
    df_split_scalar(v.h1, a.df.h1h, a.df.h1l, a.df.t1);
    df_split_scalar(v.h2, a.df.h2h, a.df.h2l, a.df.t2);
    switch (h->P) {
      case 6: launch_resident_op<OpDF<6>>(h, a, s); break;
      case 8: launch_resident_op<OpDF<8>>(h, a, s); break;
      default: launch_resident_op<OpDF<10>>(h, a, s); break;
    }
    return;
  }
  a.G = h->f64.G.ptr;
  a.B = h->f64.B.ptr;
  launch_resident_ieee<double>(h, h->f64.D.ptr, a, s);
}

template <>
void launch_resident<float>(sem_handle* h, const PcgVecs<float>& v, int iters, cudaStream_t s) {
  ResArgs<float> a{};
  resident_common(h, v, a, iters);
  a.G = h->f32.G.ptr;
  a.B = h->f32.B.ptr;
  launch_resident_ieee<float>(h, h->f32.D.ptr, a, s);
}

}  // namespace sem
