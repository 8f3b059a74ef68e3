// Even-odd line contractions in IEEE arithmetic (FP64 or FP32) for any number
// of points P per direction.
//
// D is centro-antisymmetric on GLL nodes (D_{N-i,N-l} = -D_il, and so is
// D^T), so with e_l = x_l + x_{N-l} and o_l = x_l - x_{N-l} (l < P/2) a line's
// outputs come in pairs y_i = a + s, y_{N-i} = a - s with
//   a = sum_l A_il o_l,  s = sum_l S_il e_l (+ M_iH x_H for odd P, H = P/2),
//   A_il = (M_il - M_{i,N-l}) / 2,  S_il = (M_il + M_{i,N-l}) / 2,
// and for odd P the middle output is y_H = sum_l M_Hl o_l (M_HH = 0,
// M_{H,N-l} = -M_Hl).  A line takes P^2 / 2 + 2 P operations instead of P^2.
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

// the same with x at in[off[.]] and y at out[off[.]] (in may equal out)
template <int P, class T>
__device__ __forceinline__ void eo_line(const T* in, T* out, const int (&off)[P], const T* tab) {
  T x[P];
#pragma unroll
  for (int l = 0; l < P; ++l) x[l] = in[off[l]];
  eo_dots<P, T>(x, tab, [&](int i, T y) { out[off[i]] = y; });
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
