// Pieces of the double-float element operator shared by its kernels (ax_df.cu:
// the streaming kernels; resident.cu: the grid-resident CG): the scalars, the
// shared-memory layout, the line tasks and the three-term product.
#pragma once
#include <cmath>

#include "sem_internal.cuh"
#include "df.cuh"
#include "df_tables.cuh"

namespace sem {

// D's even-odd tables as compile-time constants (df_tables.cuh, written by
// gen_df_tables.py): [t: D or D^T][A or S][high or low][i * (P/2) + l] with
// A = (M_il - M_i,N-l)/2, S = (M_il + M_i,N-l)/2, and the bounds of the
// transposed extraction dots

// h1 = m1 2^t1, h2 = m2 2^t2 with the mantissas as pairs (t = 0 while
// |h| lies in [2^-16, 2^16), see df.cuh)
struct DFScal {
  float h1h, h1l, h2h, h2l;
  int t1, t2;
};

// Shared-memory layout of one element's pairs.  P = 8: unpadded planes of 64
// pairs with rows and columns XOR-swizzled by the plane parity, position of
// (i, j, k) = 64 k + 8 (j ^ (k & 1)) + (i ^ ((j >> 1) + 4 (k & 1))): the i-, j-
// and k-lines read by the three thread groups and the per-point phases are
// all free of bank conflicts (16 threads of a half warp hit 16 distinct bank
// pairs), and an element takes 4 KB per array.  Other orders: rows padded to
// P + 2 and planes to 8 mod 16 pairs.
template <int P>
struct DFLayout {
  static constexpr int RS = P + 2;
  static constexpr int PL0 = P * RS;
  static constexpr int PL = PL0 + ((8 - (PL0 % 16)) + 16) % 16;
  static constexpr int VOL = P * PL;
  __device__ static int at(int i, int j, int k) { return k * PL + j * RS + i; }
};
template <>
struct DFLayout<8> {
  static constexpr int PL = 64;
  static constexpr int VOL = 8 * PL;
  __device__ static int at(int i, int j, int k) {
    return k * PL + 8 * (j ^ (k & 1)) + (i ^ (((j >> 1) + 4 * (k & 1)) & 7));
  }
};

// One line task: the P outputs y_i = sum_l M[i][l] x_l of the line whose
// elements sit at positions off[0..P) (M = D, or D^T when TRANS); in may equal out.
// M is centro-antisymmetric (M[N-i][N-l] = -M[i][l] on GLL nodes), so with
// e_l = x_l + x_{N-l}, o_l = x_l - x_{N-l} (l < P/2) the outputs come in pairs
// y_i = A o + S e, y_{N-i} = A o - S e with two (P/2)-term dots per pair.
template <int P, bool TRANS>
__device__ __forceinline__ void line_task(const float2* in, float2* out, const int (&off)[P]) {
  static_assert(P % 2 == 0, "even-odd split needs an even number of points");
  constexpr int H = P / 2, N = P - 1, T = TRANS ? 1 : 0;
  float xh[P], xl[P];
#pragma unroll
  for (int l = 0; l < P; ++l) {
    const float2 v = in[off[l]];
    xh[l] = v.x;
    xl[l] = v.y;
  }
  float eh[H], el[H], oh[H], ol[H];
#pragma unroll
  for (int l = 0; l < H; ++l) {
    dfadd(xh[l], xl[l], xh[N - l], xl[N - l], eh[l], el[l]);
    dfadd(xh[l], xl[l], -xh[N - l], -xl[N - l], oh[l], ol[l]);
  }
  // D annihilates constants (its rows sum to zero), hence so do the rows of S:
  // S e = sum_{l >= 1} S_il (e_l - e_0), one term fewer per dot for the
  // price of H - 1 pair subtractions.  D^T has no such property.
  constexpr int L0 = TRANS ? 0 : 1;
  if constexpr (!TRANS) {
#pragma unroll
    for (int l = 1; l < H; ++l) dfadd(eh[l], el[l], -eh[0], -el[0], eh[l], el[l]);
  }
  float yh[P], yl[P];
#pragma unroll
  for (int i = 0; i < H; ++i) {
    float Ph, Pl, Mh, Ml;
    tmac0(DFTab<P>::eo(T, 0, 0, i * H), DFTab<P>::eo(T, 0, 1, i * H), oh[0], ol[0], Ph, Pl);
    tmac0(DFTab<P>::eo(T, 1, 0, i * H + L0), DFTab<P>::eo(T, 1, 1, i * H + L0), eh[L0], el[L0], Mh,
          Ml);
#pragma unroll
    for (int l = 1; l < H; ++l)
      tmac(DFTab<P>::eo(T, 0, 0, i * H + l), DFTab<P>::eo(T, 0, 1, i * H + l), oh[l], ol[l], Ph, Pl);
#pragma unroll
    for (int l = L0 + 1; l < H; ++l)
      tmac(DFTab<P>::eo(T, 1, 0, i * H + l), DFTab<P>::eo(T, 1, 1, i * H + l), eh[l], el[l], Mh, Ml);
    dfadd(Ph, Pl, Mh, Ml, yh[i], yl[i]);
    dfadd(Ph, Pl, -Mh, -Ml, yh[N - i], yl[N - i]);
  }
#pragma unroll
  for (int i = 0; i < P; ++i) out[off[i]] = make_float2(yh[i], yl[i]);
}

// The transposed line task y_i = sum_l D_li x_l with extraction dots (df.cuh):
// the same even-odd split, with one power-of-two bound per output pair,
// sigma_i >= sum_l |A_il| |o_l| + |S_il| |e_l|.  P <= 8: the bound is taken
// from the row sums of the tables (DFTab::rb) and the largest |o| and |e| of
// the line; P = 10, whose rows are longer and whose bound that way is looser,
// forms the sum itself from the absolute entries (DFTab::ab).  Both tables
// are enlarged by 2^-18 to cover the roundings of the bound.  Both dots of a
// pair share sigma_i, so y_i = SP + SM and y_{N-i} = SP - SM are exact too.
template <int P>
__device__ __forceinline__ void line_task_xt(const float2* in, float2* out, const int (&off)[P]) {
  static_assert(P % 2 == 0, "even-odd split needs an even number of points");
  constexpr int H = P / 2, N = P - 1;
  float xh[P], xl[P];
#pragma unroll
  for (int l = 0; l < P; ++l) {
    const float2 v = in[off[l]];
    xh[l] = v.x;
    xl[l] = v.y;
  }
  float eh[H], el[H], oh[H], ol[H];
  float me = 0.0f, mo = 0.0f;
#pragma unroll
  for (int l = 0; l < H; ++l) {
    dfadd(xh[l], xl[l], xh[N - l], xl[N - l], eh[l], el[l]);
    dfadd(xh[l], xl[l], -xh[N - l], -xl[N - l], oh[l], ol[l]);
    me = fmaxf(me, fabsf(eh[l]));
    mo = fmaxf(mo, fabsf(oh[l]));
  }
#pragma unroll
  for (int i = 0; i < H; ++i) {
    float sig;
    if constexpr (P >= 10) {
      float b = 0.0f;
#pragma unroll
      for (int l = 0; l < H; ++l) {
        b = __fmaf_rn(DFTab<P>::ab(0, i * H + l), fabsf(oh[l]), b);
        b = __fmaf_rn(DFTab<P>::ab(1, i * H + l), fabsf(eh[l]), b);
      }
      sig = df_pow2_ceil(b);
    } else {
      sig = df_pow2_ceil(__fmaf_rn(DFTab<P>::rb(0, i), mo, __fmul_rn(DFTab<P>::rb(1, i), me)));
    }
    float SP, EP, SM, EM;
    xmac0(DFTab<P>::eo(1, 0, 0, i * H), DFTab<P>::eo(1, 0, 1, i * H), oh[0], ol[0], sig, SP, EP);
    xmac0(DFTab<P>::eo(1, 1, 0, i * H), DFTab<P>::eo(1, 1, 1, i * H), eh[0], el[0], sig, SM, EM);
#pragma unroll
    for (int l = 1; l < H; ++l) {
      xmac(DFTab<P>::eo(1, 0, 0, i * H + l), DFTab<P>::eo(1, 0, 1, i * H + l), oh[l], ol[l], sig, SP,
           EP);
      xmac(DFTab<P>::eo(1, 1, 0, i * H + l), DFTab<P>::eo(1, 1, 1, i * H + l), eh[l], el[l], sig, SM,
           EM);
    }
    // the line's inputs are all in registers, so the outputs may go out now
    out[off[i]] = make_float2(__fadd_rn(SP, SM), __fadd_rn(EP, EM));
    out[off[N - i]] = make_float2(__fsub_rn(SP, SM), __fsub_rn(EP, EM));
  }
}

// sum of three products g_a * v_a with extraction against sigma (df.cuh)
__device__ __forceinline__ void dot3_x(float2 g0, float2 g1, float2 g2, float2 v0, float2 v1,
                                       float2 v2, float sig, float& oh, float& ol) {
  float S, E;
  xmac0(g0.x, g0.y, v0.x, v0.y, sig, S, E);
  xmac(g1.x, g1.y, v1.x, v1.y, sig, S, E);
  xmac(g2.x, g2.y, v2.x, v2.y, sig, S, E);
  oh = S;
  ol = E;
}

// h = m 2^t with t = df_pick_exp(|h|) and m as a pair (exact: m is h times a
// power of two, split into its leading 24 bits and the next 24)
inline void df_split_scalar(double h, float& hi, float& lo, int& t) {
  t = df_pick_exp(std::fabs(h));
  const double m = std::ldexp(h, -t);
  hi = (float)m;
  lo = (float)(m - (double)hi);
}

}  // namespace sem
