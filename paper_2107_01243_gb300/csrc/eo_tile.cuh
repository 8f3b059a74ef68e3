// Line contractions y = D x and y = D^T x in IEEE arithmetic (FP64 or FP32) for
// any number of points P per direction, with D's entries or its even-odd split.
//
// D is centro-antisymmetric on GLL nodes (D_{N-i,N-l} = -D_il, and so is
// D^T), so with e_l = x_l + x_{N-l} and o_l = x_l - x_{N-l} (l < P/2) a line's
// outputs come in pairs y_i = a + s, y_{N-i} = a - s with
//   a = sum_l A_il o_l,  s = sum_l S_il e_l (+ M_iH x_H for odd P, H = P/2),
//   A_il = (M_il - M_{i,N-l}) / 2,  S_il = (M_il + M_{i,N-l}) / 2,
// and for odd P the middle output is y_H = sum_l M_Hl o_l (M_HH = 0,
// M_{H,N-l} = -M_Hl).  A line takes P^2 / 2 + 2 P operations instead of P^2, but
// on smooth lines it rounds worse (e_l rounds at twice the size of x before the
// large terms cancel): RMS error of the element operator against 128 bits, N = 6,
// on random / smooth / nearly constant fields 0.84 / 2.4 / 3.5 times that of plain
// dot products.  A mixed solve on flat elements whose FP64 residual took the split
// stood at 1.5e-12 of b (N = 4) and 1.03e-12 (N = 6), with plain lines at 0.97e-12
// and 0.87e-12.  So the lines take D's entries, but for IEEE FP64 at P = 8 and 10,
// whose results have always been the split's (2.6% and 17% less time there).
#pragma once
#include "sem_internal.cuh"

namespace sem {

// table of one matrix M: [A: H x H][S: H x HS][middle row: H, odd P], HS = H
// for even P and H + 1 (with the middle column) for odd P
template <int P>
struct EoTab {
  static constexpr int H = P / 2, ODD = P % 2, HS = H + ODD;
  static constexpr int A = 0, S = H * H, M = H * H + H * HS;
  static constexpr int SIZE = M + ODD * H;
};

// whether the lines of this order and precision take the split, and the table of
// one such line kernel in shared memory: the two even-odd tables, or D row-major
constexpr bool eo_split(int P, bool f64) { return f64 && (P == 8 || P == 10); }
template <int P, class T>
struct LineTab {
  static constexpr bool EO = eo_split(P, sizeof(T) == 8);
  static constexpr int SIZE = EO ? 2 * EoTab<P>::SIZE : P * P;
  static constexpr int FROM = EO ? P * P : 0;       // its place in OpData::D
};

// y = M x for a line in registers; put(i, y_i) receives the outputs.  tab in
// shared memory (one broadcast read per use: the compiler would otherwise
// keep the whole table in registers across the element loop)
template <int P, class T, class PUT>
__device__ __forceinline__ void eo_dots(const T (&x)[P], const T* tab, PUT put) {
  using E = EoTab<P>;
  constexpr int H = E::H, HS = E::HS, N = P - 1;
  T e[HS], o[H];
#pragma unroll
  for (int l = 0; l < H; ++l) {
    e[l] = x[l] + x[N - l];
    o[l] = x[l] - x[N - l];
  }
  if constexpr (E::ODD) e[H] = x[H];
#pragma unroll
  for (int i = 0; i < H; ++i) {
    T a = tab[E::A + i * H] * o[0];
    T s = tab[E::S + i * HS] * e[0];
#pragma unroll
    for (int l = 1; l < HS; ++l) {
      if (l < H) a = fma(tab[E::A + i * H + l], o[l], a);
      s = fma(tab[E::S + i * HS + l], e[l], s);
    }
    put(i, a + s);
    put(N - i, a - s);
  }
  if constexpr (E::ODD) {
    T a = tab[E::M] * o[0];
#pragma unroll
    for (int l = 1; l < H; ++l) a = fma(tab[E::M + l], o[l], a);
    put(H, a);
  }
}

// y = D x, or D^T x (TRANS), with x at in[off[.]] and y at out[off[.]] (in may
// equal out); tab: LineTab in shared memory
template <int P, class T, bool TRANS>
__device__ __forceinline__ void tab_line(const T* in, T* out, const int (&off)[P], const T* tab) {
  T x[P];
#pragma unroll
  for (int l = 0; l < P; ++l) x[l] = in[off[l]];
  if constexpr (LineTab<P, T>::EO) {
    eo_dots<P, T>(x, tab + (TRANS ? EoTab<P>::SIZE : 0), [&](int i, T y) { out[off[i]] = y; });
  } else {
#pragma unroll
    for (int i = 0; i < P; ++i) {
      T y = tab[TRANS ? i : i * P] * x[0];
#pragma unroll
      for (int l = 1; l < P; ++l) y = fma(tab[TRANS ? l * P + i : i * P + l], x[l], y);
      out[off[i]] = y;
    }
  }
}

// host: the tables of D and D^T, one after the other (2 EoTab<P>::SIZE values)
inline std::vector<double> eo_tables(int P, const std::vector<double>& D) {
  const int H = P / 2, odd = P % 2, HS = H + odd, N = P - 1;
  std::vector<double> out;
  for (int t = 0; t < 2; ++t) {
    auto M = [&](int i, int l) { return t ? D[l * P + i] : D[i * P + l]; };
    for (int i = 0; i < H; ++i)
      for (int l = 0; l < H; ++l) out.push_back(0.5 * (M(i, l) - M(i, N - l)));
    for (int i = 0; i < H; ++i)
      for (int l = 0; l < HS; ++l)
        out.push_back(l < H ? 0.5 * (M(i, l) + M(i, N - l)) : M(i, H));
    if (odd)
      for (int l = 0; l < H; ++l) out.push_back(M(H, l));
  }
  return out;
}

// shared-memory position of (i, j, k).  8-byte values: P = 8 uses unpadded
// 64-value planes with rows and columns XOR-swizzled by the plane parity (the
// lines of all three directions and the point phases are free of bank
// conflicts); other orders pad rows to P + 2 (even P) and planes to 8 mod 16
// values.  4-byte values: rows padded to an odd length.
template <int P, class T>
struct EoLayout {
  static constexpr int RS = sizeof(T) == 8 ? (P % 2 ? P : P + 2) : (P | 1);
  static constexpr int PL0 = P * RS;
  static constexpr int PL = sizeof(T) == 8 ? PL0 + ((8 - (PL0 % 16)) + 16) % 16 : PL0;
  static constexpr int VOL = P * PL;
  __device__ static int at(int i, int j, int k) { return k * PL + j * RS + i; }
};
template <>
struct EoLayout<8, double> {
  static constexpr int PL = 64;
  static constexpr int VOL = 8 * PL;
  __device__ static int at(int i, int j, int k) {
    return k * PL + 8 * (j ^ (k & 1)) + (i ^ (((j >> 1) + 4 * (k & 1)) & 7));
  }
};

}  // namespace sem
