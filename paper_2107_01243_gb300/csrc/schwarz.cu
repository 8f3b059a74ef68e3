// Two-level additive overlapping Schwarz preconditioner (arXiv 2107.01243 §4:
// Neko's pressure preconditioner, M^-1 = R_0^T A_0^-1 R_0 + sum_k R_k^T
// A~_k^-1 R_k, after Nek5000), applied in FP32:
//
// local level   subdomain = element grown by one GLL point into each
//               neighbour, (N + 3)^3 lattice points without points outside
//               the box and without Dirichlet points.  A~_e is the separable
//               Kronecker sum of 1D spectral-element stiffness and mass
//               matrices of the element and its neighbours (undeformed box
//               spacing), inverted by fast diagonalisation: per direction
//               A S = B S diag(lam), S^T B S = I, computed once on the host.
//               One CTA per element: gather the grown box of r from the global
//               vector by columns, S^T along z, then x, then y with the diagonal
//               scaling and S back, S along x and z, scatter-add to z by L2
//               reductions.  The same kernel forms the coarse restriction from
//               the element's own points.
// coarse level  trilinear vertex functions; A_0 = R_0 H R_0^T assembled from
//               8 x 8 element matrices Phi^T H_e Phi (computed at setup with
//               the FP64 element operator, stored packed in FP32), as a
//               27-point stencil where the vertices fit one launch; a fixed
//               number of Jacobi-PCG iterations from zero: in one cluster
//               (up to 16,384 vertices), in one cooperative grid, or with the
//               FP32 CG steps of cg.cu and an element-by-element matvec.
// output        z_L = mask o (z_local[g(L)] + R_0^T c) as FP64 L-vector.
#include <cmath>
#include <memory>
#include <vector>

#include "sem_internal.cuh"
#include "grid_dots.cuh"
#include "reduce.cuh"
#include "tma.cuh"

namespace sem {
namespace {

// threads of the local-solve CTA: one per z-column of the grown box, whole warps
template <int PE>
struct SwCfg {
  static constexpr int THREADS = PE * PE <= 128 ? 128 : (PE * PE + 31) / 32 * 32;
  static constexpr int MINB = PE * PE <= 128 ? 6 : 4;
};
constexpr int kNbr = 0, kDir = 1, kFree = 2;

// ------------------------------------------------------------------ host setup
// Symmetric eigen-decomposition by cyclic Jacobi rotations (n <= 13):
// A = V diag(lam) V^T, V orthogonal (columns are eigenvectors).
void jacobi_eigen(int n, std::vector<double> A, std::vector<double>& V, std::vector<double>& lam) {
  V.assign(n * n, 0.0);
  for (int i = 0; i < n; ++i) V[i * n + i] = 1.0;
  double scale = 0.0;
  for (double a : A) scale = std::max(scale, std::fabs(a));
  for (int sweep = 0; sweep < 100; ++sweep) {
    double off = 0.0;
    for (int p = 0; p < n; ++p)
      for (int q = p + 1; q < n; ++q) off = std::max(off, std::fabs(A[p * n + q]));
    if (off <= 1e-16 * scale) break;
    for (int p = 0; p < n; ++p) {
      for (int q = p + 1; q < n; ++q) {
        const double apq = A[p * n + q];
        if (std::fabs(apq) <= 1e-300) continue;
        const double theta = (A[q * n + q] - A[p * n + p]) / (2.0 * apq);
        const double t = (theta >= 0 ? 1.0 : -1.0) / (std::fabs(theta) + std::sqrt(theta * theta + 1.0));
        const double c = 1.0 / std::sqrt(t * t + 1.0), s = t * c;
        for (int k = 0; k < n; ++k) {           // columns p, q
          const double akp = A[k * n + p], akq = A[k * n + q];
          A[k * n + p] = c * akp - s * akq;
          A[k * n + q] = s * akp + c * akq;
        }
        for (int k = 0; k < n; ++k) {           // rows p, q
          const double apk = A[p * n + k], aqk = A[q * n + k];
          A[p * n + k] = c * apk - s * aqk;
          A[q * n + k] = s * apk + c * aqk;
        }
        for (int k = 0; k < n; ++k) {
          const double vkp = V[k * n + p], vkq = V[k * n + q];
          V[k * n + p] = c * vkp - s * vkq;
          V[k * n + q] = s * vkp + c * vkq;
        }
      }
    }
  }
  lam.resize(n);
  for (int i = 0; i < n; ++i) lam[i] = A[i * n + i];
}

// 1D stiffness and lumped mass on the N + 3 points of a grown element
// (position a = lattice point N e - 1 + a), from the element and its
// neighbours of length L; positions not kept are decoupled (unit diagonal).
void extended_1d(const sem_handle* h, double L, int lo, int hi, std::vector<double>& A,
                 std::vector<double>& B, unsigned& keep) {
  const int N = h->N, P = h->P, Pe = N + 3, n3 = 3 * N + 1;
  std::vector<double> ae(P * P, 0.0);
  for (int i = 0; i < P; ++i)
    for (int j = 0; j < P; ++j) {
      double acc = 0.0;
      for (int k = 0; k < P; ++k) acc += h->Dh[k * P + i] * h->wq[k] * h->Dh[k * P + j];
      ae[i * P + j] = (2.0 / L) * acc;
    }
  std::vector<double> A3(n3 * n3, 0.0), B3(n3, 0.0);
  for (int m = 0; m < 3; ++m) {
    if ((m == 0 && lo != kNbr) || (m == 2 && hi != kNbr)) continue;
    const int s0 = m * N;
    for (int i = 0; i < P; ++i) {
      B3[s0 + i] += 0.5 * L * h->wq[i];
      for (int j = 0; j < P; ++j) A3[(s0 + i) * n3 + s0 + j] += ae[i * P + j];
    }
  }
  keep = (1u << Pe) - 1u;
  if (lo != kNbr) {
    keep &= ~1u;
    if (lo == kDir) keep &= ~2u;
  }
  if (hi != kNbr) {
    keep &= ~(1u << (N + 2));
    if (hi == kDir) keep &= ~(1u << (N + 1));
  }
  A.assign(Pe * Pe, 0.0);
  B.assign(Pe, 0.0);
  for (int a = 0; a < Pe; ++a) {
    const int ga = N - 1 + a;
    B[a] = B3[ga];
    for (int b = 0; b < Pe; ++b) A[a * Pe + b] = A3[ga * n3 + N - 1 + b];
  }
  for (int a = 0; a < Pe; ++a) {
    if (keep & (1u << a)) continue;
    for (int b = 0; b < Pe; ++b) {
      A[a * Pe + b] = 0.0;
      A[b * Pe + a] = 0.0;
    }
    A[a * Pe + a] = 1.0;
    B[a] = 1.0;
  }
}

// ------------------------------------------------------------------ device tables
// Per direction d and element kind v (bit 0: first along d, bit 1: last),
// rows padded to R floats: ST[a'][a] = S[a][a'], then S[a][a'], then lam[a].
template <int PE>
struct SwLayout {
  static constexpr int R = (PE + 3) / 4 * 4;
  static constexpr int TAB = 2 * PE * R + R;         // one (d, v) table
  static constexpr int ALL = 12 * TAB;               // then h1 (lx + ly + lz) + h2 of the
                                                     // interior element, [c][b][a]
};

struct SwParams {
  int N, nelx, nely, nelz, gx, gy;
  long long sk;
  FastDiv dnx, dny;
  unsigned keep[3][4];
  float h1, h2;
  int do_local, do_coarse;
  float phi[2][kMaxP];                 // trilinear vertex functions at the GLL nodes
};

template <int R>
__device__ __forceinline__ float dot_row(const float* __restrict__ row, const float (&x)[R], int n) {
  float acc = 0.0f;
#pragma unroll
  for (int a = 0; a < R; a += 4) {
    const float4 v = *reinterpret_cast<const float4*>(row + a);
    if (a + 0 < n) acc = fmaf(v.x, x[a + 0], acc);
    if (a + 1 < n) acc = fmaf(v.y, x[a + 1], acc);
    if (a + 2 < n) acc = fmaf(v.z, x[a + 2], acc);
    if (a + 3 < n) acc = fmaf(v.w, x[a + 3], acc);
  }
  return acc;
}

// S of the interior elements (kind 0) per direction, [a][a'], in the kernel
// parameters: constant-bank operands of the line tasks
template <int PE>
struct SwConst {
  float S[3][PE * PE];
};

// y = S^T x (TRANS) or S x along direction DIR; interior kinds from the constant
// bank, the others from the table tb of SwLayout in shared memory
template <int PE, int DIR, bool TRANS, class PUT>
__device__ __forceinline__ void sw_line(const SwConst<PE>& k, bool interior, const float* tb,
                                        const float (&x)[SwLayout<PE>::R], PUT put) {
  constexpr int R = SwLayout<PE>::R;
  if (interior) {
#pragma unroll
    for (int i = 0; i < PE; ++i) {
      float y = (TRANS ? k.S[DIR][i] : k.S[DIR][i * PE]) * x[0];
#pragma unroll
      for (int l = 1; l < PE; ++l)
        y = fmaf(TRANS ? k.S[DIR][l * PE + i] : k.S[DIR][i * PE + l], x[l], y);
      put(i, y);
    }
  } else {
    const float* t = tb + (TRANS ? 0 : PE * R);
#pragma unroll
    for (int i = 0; i < PE; ++i) put(i, dot_row<R>(t + i * R, x, PE));
  }
}

// One element per CTA.  Thread (a, b) < PE^2 owns the z-column of the grown box:
// it gathers the column, applies S^T along z in registers and writes
// box[c][b][a] (rows padded to R, moved as 16-byte vectors); the x- and
// y-directions run as line tasks through shared memory (S^T along x; along y
// S^T, the diagonal scaling and S; S along x); the thread then reads its column
// back, applies S along z in registers and adds the kept points to z.  Factors
// along different directions commute, so this order gives the same A~^-1 as x,
// y, z first.  The coarse restriction is taken from the gathered columns of the
// element's own points (a, b, c in 1 .. P): z-weighted sums per column, then
// the last warp, which has the fewest lines, adds them up.
// The kernel is bound by issue and by the latency of its line phases: S as
// constant operands (an interior direction reads no table: the persistent form
// with all tables in shared memory spent three 16-byte reads on every output),
// the interior scaling's divisors as a table, and one element a CTA, so
// that tables that are not used are not loaded and the registers allow twice
// the CTAs.  13,824 elements, N = 7: 95 us (160 before; 91 with reciprocals in the
// table, a rounding more).
template <int PE>
__global__ void __launch_bounds__(SwCfg<PE>::THREADS, SwCfg<PE>::MINB)
schwarz_local_kernel(const float* __restrict__ rg, float* __restrict__ zg,
                     float* __restrict__ rc, const float* __restrict__ tab_g,
                     const __grid_constant__ SwParams prm,
                     const __grid_constant__ SwConst<PE> kst) {
  using L = SwLayout<PE>;
  constexpr int R = L::R, P = PE - 2, N = PE - 3, T = SwCfg<PE>::THREADS, PE2 = PE * PE;
  static_assert(PE2 <= T, "a line per thread");
  __shared__ __align__(16) float tab[3][L::TAB];
  __shared__ __align__(16) float box[PE2 * R];
  __shared__ float cs[2][PE2];
  const int tid = threadIdx.x, e = blockIdx.x;
  const bool owner = tid < PE2;
  const int ca = tid % PE, cb = tid / PE;          // this thread's column (a, b)
  const uint32_t r1 = prm.dnx.div((uint32_t)e);
  const int ex = e - (int)r1 * prm.nelx;
  const uint32_t q1 = prm.dny.div(r1);
  const int ey = (int)(r1 - q1 * (uint32_t)prm.nely), ez = (int)q1;
  const int vk[3] = {(ex == 0 ? 1 : 0) | (ex == prm.nelx - 1 ? 2 : 0),
                     (ey == 0 ? 1 : 0) | (ey == prm.nely - 1 ? 2 : 0),
                     (ez == 0 ? 1 : 0) | (ez == prm.nelz - 1 ? 2 : 0)};
  const unsigned kx = prm.keep[0][vk[0]], ky = prm.keep[1][vk[1]], kz = prm.keep[2][vk[2]];
  const bool colkeep = owner && ((kx >> ca) & 1u) && ((ky >> cb) & 1u);
  // lattice index of (a, b, 0) of this thread's column
  const long long cbase = (long long)(N * ex - 1 + ca) + (long long)prm.gx * (N * ey - 1 + cb) +
                          prm.sk * (long long)(N * ez - 1);
  float col[R];
#pragma unroll
  for (int c = 0; c < R; ++c)
    col[c] = (c < PE && colkeep && ((kz >> c) & 1u)) ? __ldg(rg + cbase + prm.sk * c) : 0.0f;
  // the tables of the directions that are not interior; the eigenvalues unless
  // the whole element is interior (then the divisors serve)
  const bool inner = (vk[0] | vk[1] | vk[2]) == 0;
  if (!inner) {
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const float* src = tab_g + (d * 4 + vk[d]) * L::TAB;
      for (int q = tid + (vk[d] ? 0 : 2 * PE * R); q < L::TAB; q += T) tab[d][q] = __ldg(src + q);
    }
  }
  if (prm.do_coarse && owner) {
    float s0 = 0.0f, s1 = 0.0f;
    if (ca >= 1 && ca <= P && cb >= 1 && cb <= P) {
      const int i = ca - 1, j = cb - 1;
      const float mij = ((i == 0 && ex > 0) || (i == N && ex < prm.nelx - 1) ? 0.5f : 1.0f) *
                        ((j == 0 && ey > 0) || (j == N && ey < prm.nely - 1) ? 0.5f : 1.0f);
#pragma unroll
      for (int k = 0; k < P; ++k) {
        const float mk = (k == 0 && ez > 0) || (k == N && ez < prm.nelz - 1) ? 0.5f : 1.0f;
        const float rv = mk * col[k + 1];
        s0 = fmaf(prm.phi[0][k], rv, s0);
        s1 = fmaf(prm.phi[1][k], rv, s1);
      }
      s0 *= mij;
      s1 *= mij;
    }
    cs[0][tid] = s0;
    cs[1][tid] = s1;
  }
  __syncthreads();
  if (prm.do_local && owner)               // S^T along z in registers, to the box
    sw_line<PE, 2, true>(kst, vk[2] == 0, tab[2], col,
                         [&](int c, float y) { box[(c * PE + cb) * R + ca] = y; });
  if (prm.do_coarse && tid >= T - 32) {    // the eight vertex sums of this element
    const int lane = tid & 31;
    float acc[8];
#pragma unroll
    for (int v = 0; v < 8; ++v) acc[v] = 0.0f;
    for (int q = lane; q < P * P; q += 32) {
      const int i = q % P, j = q / P, at = (j + 1) * PE + i + 1;
      const float s0 = cs[0][at], s1 = cs[1][at];
#pragma unroll
      for (int v = 0; v < 8; ++v)
        acc[v] = fmaf(prm.phi[v & 1][i] * prm.phi[(v >> 1) & 1][j], (v >> 2) ? s1 : s0, acc[v]);
    }
#pragma unroll
    for (int v = 0; v < 8; ++v)
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) acc[v] += __shfl_xor_sync(0xffffffffu, acc[v], o);
    float mine = acc[0];
#pragma unroll
    for (int v = 1; v < 8; ++v) mine = lane == v ? acc[v] : mine;
    if (lane < 8) {
      const long long vi = (long long)(ex + (lane & 1)) +
                           (long long)(prm.nelx + 1) *
                               ((ey + ((lane >> 1) & 1)) + (long long)(prm.nely + 1) * (ez + (lane >> 2)));
      red_add(rc + vi, mine);
    }
  }
  if (!prm.do_local) return;
  __syncthreads();
  float x[R], y[R];
  float4* row = reinterpret_cast<float4*>(box + tid * R);
  auto row_in = [&]() {
#pragma unroll
    for (int a = 0; a < R; a += 4) {
      const float4 v = row[a / 4];
      x[a] = v.x; x[a + 1] = v.y; x[a + 2] = v.z; x[a + 3] = v.w;
    }
  };
  auto row_out = [&]() {
#pragma unroll
    for (int a = 0; a < R; a += 4) row[a / 4] = make_float4(y[a], y[a + 1], y[a + 2], y[a + 3]);
  };
#pragma unroll
  for (int a = 0; a < R; ++a) y[a] = 0.0f;
  if (owner) {                             // S^T along x on line (b, c)
    row_in();
    sw_line<PE, 0, true>(kst, vk[0] == 0, tab[0], x, [&](int a, float v) { y[a] = v; });
    row_out();
  }
  __syncthreads();
  if (owner) {                             // along y on line (a, c): S^T, scaling, S
    float* yl = box + cb * PE * R + ca;    // (a, c) = (tid % PE, tid / PE)
#pragma unroll
    for (int b = 0; b < R; ++b) x[b] = b < PE ? yl[b * R] : 0.0f;
    sw_line<PE, 1, true>(kst, vk[1] == 0, tab[1], x, [&](int b, float v) { y[b] = v; });
    if (inner) {
      const float* den = tab_g + L::ALL + cb * PE2 + ca;     // h1 (lx + ly + lz) + h2
#pragma unroll
      for (int b = 0; b < PE; ++b) y[b] /= __ldg(den + b * PE);
    } else {
      const float lac = tab[0][2 * PE * R + ca] + tab[2][2 * PE * R + cb];
#pragma unroll
      for (int b = 0; b < PE; ++b) y[b] /= prm.h1 * (lac + tab[1][2 * PE * R + b]) + prm.h2;
    }
    sw_line<PE, 1, false>(kst, vk[1] == 0, tab[1], y, [&](int b, float v) { yl[b * R] = v; });
  }
  __syncthreads();
  if (owner) {                             // S along x
    row_in();
#pragma unroll
    for (int a = 0; a < R; ++a) y[a] = 0.0f;
    sw_line<PE, 0, false>(kst, vk[0] == 0, tab[0], x, [&](int a, float v) { y[a] = v; });
    row_out();
  }
  __syncthreads();
  if (colkeep) {                           // S along z in registers, add the kept points
#pragma unroll
    for (int c = 0; c < R; ++c) x[c] = c < PE ? box[(c * PE + cb) * R + ca] : 0.0f;
    sw_line<PE, 2, false>(kst, vk[2] == 0, tab[2], x, [&](int c, float v) {
      if ((kz >> c) & 1u) red_add(zg + cbase + prm.sk * c, v);
    });
  }
}

// packed index of (r, c), r <= c, in the upper triangle of an 8 x 8 matrix
__host__ __device__ constexpr int pk(int r, int c) { return r * 8 - r * (r - 1) / 2 + (c - r); }

// w += A_0 p element by element (K packed symmetric, FP32)
__global__ void k_coarse_matvec(int E, const float* __restrict__ K, const float* __restrict__ p,
                                float* __restrict__ w, int nelx, int nely, FastDiv dnx,
                                FastDiv dny) {
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < E; e += gridDim.x * blockDim.x) {
    const uint32_t r1 = dnx.div((uint32_t)e);
    const int ex = e - (int)r1 * nelx;
    const uint32_t q1 = dny.div(r1);
    const int ey = (int)(r1 - q1 * (uint32_t)nely), ez = (int)q1;
    int vi[8];
    float pv[8];
#pragma unroll
    for (int v = 0; v < 8; ++v) {
      vi[v] = (ex + (v & 1)) + (nelx + 1) * ((ey + ((v >> 1) & 1)) + (nely + 1) * (ez + (v >> 2)));
      pv[v] = p[vi[v]];
    }
    const float* Ke = K + (size_t)e * 36;
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      float acc = 0.0f;
#pragma unroll
      for (int c = 0; c < 8; ++c) acc = fmaf(Ke[r <= c ? pk(r, c) : pk(c, r)], pv[c], acc);
      red_add(w + vi[r], acc);
    }
  }
}

// ------------------------------------------------------------------ coarse CG in one launch
// A_0 as a 27-point stencil on the vertices: st[o][v] = sum of the entries of
// the elements that hold both v and its neighbour o (dx, dy, dz in {-1, 0, 1},
// o = (dx + 1) + 3 (dy + 1) + 9 (dz + 1)); neighbours outside the box get 0.
__global__ void k_coarse_stencil(int nelx, int nely, int nelz, const float* __restrict__ K,
                                 float* __restrict__ st, int nv) {
  const int nvx = nelx + 1, nvy = nely + 1;
  for (int v = blockIdx.x * blockDim.x + threadIdx.x; v < nv; v += gridDim.x * blockDim.x) {
    const int x = v % nvx, y = (v / nvx) % nvy, z = v / (nvx * nvy);
    for (int o = 0; o < 27; ++o) {
      const int dx = o % 3 - 1, dy = (o / 3) % 3 - 1, dz = o / 9 - 1;
      double acc = 0.0;
      for (int c = 0; c < 8; ++c) {            // v is corner c of the element at (ex, ey, ez)
        const int cx = c & 1, cy = (c >> 1) & 1, cz = c >> 2;
        const int ex = x - cx, ey = y - cy, ez = z - cz;
        const int bx = cx + dx, by = cy + dy, bz = cz + dz;   // the neighbour's corner
        if (ex < 0 || ex >= nelx || ey < 0 || ey >= nely || ez < 0 || ez >= nelz) continue;
        if (bx < 0 || bx > 1 || by < 0 || by > 1 || bz < 0 || bz > 1) continue;
        const int b = bx + 2 * by + 4 * bz;
        const size_t e = (size_t)ex + (size_t)nelx * (ey + (size_t)nely * ez);
        acc += (double)K[e * 36 + (c <= b ? pk(c, b) : pk(b, c))];
      }
      st[(size_t)o * nv + v] = (float)acc;
    }
  }
}

constexpr int kCoarseThreads = 256;
constexpr int kCoarseBlocks = 608;   // the most CTAs (their sums fit the shared memory)

struct CoarseArgs {
  const float *st, *dinv, *r;       // stencil, Jacobi inverse (0: masked), right-hand side
  float *x, *p0, *p1, *z;           // solution; directions (two buffers), residual scaled
  longlong2* partials;              // 2 gridDim.x values, taken in turn
  unsigned* bar;                    // zero at launch
  int* err;
  uint64_t timeout_ns;
  int nvx, nvy, nvz, iters;
};

// iters Jacobi-CG iterations from zero, a thread per vertex with its stencil
// row, x, r and dinv in registers (a cooperative launch; two grid barriers an
// iteration).  A thread forms its neighbours' p = z + beta p_old itself, so that
// the barrier that gives beta needs none after it.  Ten iterations on 25^3
// vertices took 240 us as 40 launches of a few microseconds each.
__global__ void __launch_bounds__(kCoarseThreads)
k_coarse_cg(const __grid_constant__ CoarseArgs a) {
  constexpr int NW = kCoarseThreads / 32;
  extern __shared__ longlong2 sp[];
  __shared__ FxVal s_w[2][16];
  __shared__ double s_tot[2], s_rz;
  __shared__ float s_alpha, s_beta;
  __shared__ int s_bad, s_stop;
  const int nv = a.nvx * a.nvy * a.nvz;
  const int v = blockIdx.x * kCoarseThreads + threadIdx.x;
  const bool act = v < nv;
  const int x0 = act ? v % a.nvx : 0, y0 = act ? (v / a.nvx) % a.nvy : 0,
            z0 = act ? v / (a.nvx * a.nvy) : 0;
  float c[27];
#pragma unroll
  for (int o = 0; o < 27; ++o) c[o] = act ? __ldg(a.st + (size_t)o * nv + v) : 0.0f;
  const float d = act ? a.dinv[v] : 0.0f;
  float r = act ? a.r[v] : 0.0f, x = 0.0f, z = d * r, p = 0.0f;
  if (act) {
    __stcg(a.z + v, z);
    __stcg(a.p0 + v, 0.0f);
  }
  if (threadIdx.x == 0) {
    s_bad = 0;
    s_stop = 0;
  }
  // a wait ran out (recorded in err): no earlier call's solution is left in x
  auto give_up = [&] {
    if (act) a.x[v] = __int_as_float(0x7FC00000);
  };
  unsigned met = 0;
  float *pold = a.p0, *pnew = a.p1;
  {
    const double v0[1] = {fx_prod(r, z)};
    met += gridDim.x;
    if (!grid_dots<1, NW>(v0, s_w, sp, s_tot, a.partials + gridDim.x, a.bar, met, a.err, a.timeout_ns, &s_bad,
                          [&] {
                            s_rz = s_tot[0];
                            s_beta = 0.0f;
                            s_stop = dbits(s_tot[0]) <= 0 || is_nan(s_tot[0]);
                          }))
      return give_up();
  }
  for (int it = 0; it < a.iters && !s_stop; ++it) {
    const float beta = s_beta;
    float w = 0.0f;
    p = fmaf(beta, p, z);
    if (act) {
      __stcg(pnew + v, p);
#pragma unroll
      for (int o = 0; o < 27; ++o) {
        const int dx = o % 3 - 1, dy = (o / 3) % 3 - 1, dz = o / 9 - 1;
        if (o == 13) {
          w = fmaf(c[13], p, w);
        } else if (x0 + dx >= 0 && x0 + dx < a.nvx && y0 + dy >= 0 && y0 + dy < a.nvy &&
                   z0 + dz >= 0 && z0 + dz < a.nvz) {
          const int n = v + dx + a.nvx * (dy + a.nvy * dz);
          w = fmaf(c[o], fmaf(beta, __ldcg(pold + n), __ldcg(a.z + n)), w);
        }
      }
    }
    const double v1[1] = {fx_prod(p, w)};
    met += gridDim.x;
    if (!grid_dots<1, NW>(v1, s_w, sp, s_tot, a.partials, a.bar, met, a.err, a.timeout_ns, &s_bad,
                          [&] {
                            s_stop = dbits(s_tot[0]) <= 0 || is_nan(s_tot[0]);
                            s_alpha = s_stop ? 0.0f : (float)(s_rz / s_tot[0]);
                          }))
      return give_up();
    if (s_stop) break;
    x = fmaf(s_alpha, p, x);
    r = fmaf(-s_alpha, w, r);
    z = d * r;
    if (it + 1 == a.iters) break;            // the last direction has been taken
    if (act) __stcg(a.z + v, z);
    const double v2[1] = {fx_prod(r, z)};
    met += gridDim.x;
    if (!grid_dots<1, NW>(v2, s_w, sp, s_tot, a.partials + gridDim.x, a.bar, met, a.err,
                          a.timeout_ns, &s_bad, [&] {
                            s_stop = dbits(s_tot[0]) <= 0 || is_nan(s_tot[0]);
                            s_beta = s_stop ? 0.0f : (float)(s_tot[0] / s_rz);
                            s_rz = s_tot[0];
                          }))
      return give_up();
    float* t = pold;
    pold = pnew;
    pnew = t;
  }
  if (act) a.x[v] = x;
}

// ---- the same iterations in one cluster of 16 CTAs, where a thread per vertex
// fits (up to 16,384 vertices): barriers and sums through distributed shared
// memory instead of the grid's global ones.  A CTA keeps p of its own vertices
// and of their neighbours (a halo of one layer and row on either side) in shared
// memory.  Bound by the latency of its 20 sums, one after another: 10
// iterations on 25^3 vertices 50 us (57 with the products formed in FP64, 97 as a
// cooperative grid).
constexpr int kClusterCtas = 16, kClusterThreads = 1024;

__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_barrier() {
  asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::
                   : "memory");
}
// 16 bytes to the same shared address of CTA `to` of the cluster
__device__ __forceinline__ void cluster_put(longlong2* p, uint32_t to, longlong2 v) {
  uint32_t a;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(smem_addr(p)), "r"(to));
  asm volatile("st.shared::cluster.v2.s64 [%0], {%1, %2};" ::"r"(a), "l"(v.x), "l"(v.y) : "memory");
}

// Sum of v over the cluster, in every thread of warp 0 (others get nothing).
// slots: kClusterCtas entries, two sets used in turn by the caller.
__device__ __forceinline__ double cluster_sum(double v, FxVal* sw, longlong2* slots) {
  constexpr int NW = kClusterThreads / 32;
  const int lane = threadIdx.x & 31;
  const FxVal f = fx_warp_sum(v);
  if (lane == 0) sw[threadIdx.x >> 5] = f;
  __syncthreads();
  if (threadIdx.x < 32) {
    const FxTot t = fx_lane_sum(sw[lane]);   // NW = 32 warps: at most 32 x 2^62
    if (lane < kClusterCtas) cluster_put(slots + cluster_rank(), lane, fx_pack(t, 5));
    __syncwarp();
  }
  static_assert(NW == 32, "a lane per warp");
  cluster_barrier();
  if (threadIdx.x >= 32) return 0.0;
  const longlong2 p = lane < kClusterCtas ? slots[lane] : make_longlong2(0, 1);
  const FxTot t = fx_lane_sum(FxVal{p.x, (int)p.y});
  return fx_round(t.acc.hi, t.acc.lo, t.e);
}

// a / b rounded to FP32, for positive normal doubles and infinities (an FP64 division takes a
// lone warp half a microsecond): the significands as pairs of floats, the
// quotient of the leading parts and its first-order correction (Dekker 1971)
__device__ __forceinline__ float ratio32(double a, double b) {
  const long long ia = dbits(a), ib = dbits(b);
  if (max(ia, ib) >= 0x7FF0000000000000ll) return (float)(a / b);
  const long long ma = (ia & 0xFFFFFFFFFFFFFll) | (1ll << 52);
  const long long mb = (ib & 0xFFFFFFFFFFFFFll) | (1ll << 52);
  const float ah = (float)(int)(ma >> 29), al = (float)(int)(ma & 0x1FFFFFFF) * 0x1p-29f;
  const float bh = (float)(int)(mb >> 29), bl = (float)(int)(mb & 0x1FFFFFFF) * 0x1p-29f;
  const float q = __fdiv_rn(ah, bh);
  const float rem = fmaf(-q, bl, fmaf(-q, bh, ah) + al);
  return ldexpf(q + __fdiv_rn(rem, bh), (int)(ia >> 52) - (int)(ib >> 52));
}

__global__ void __launch_bounds__(kClusterThreads, 1)
k_coarse_cluster(const __grid_constant__ CoarseArgs a, int nvc, int halo) {
  extern __shared__ float s_p[];             // p of vertices v0 - halo .. v0 + nvc + halo
  __shared__ FxVal sw[32];
  __shared__ longlong2 slots[2][kClusterCtas];
  __shared__ float s_coef;                   // alpha or beta of the step
  __shared__ int s_stop;
  const int nv = a.nvx * a.nvy * a.nvz, tid = threadIdx.x;
  const int v0 = (int)cluster_rank() * nvc, v = v0 + tid;
  const bool act = tid < nvc && v < nv;
  float c[27];
#pragma unroll
  for (int o = 0; o < 27; ++o) c[o] = act ? __ldg(a.st + (size_t)o * nv + v) : 0.0f;
  const float d = act ? a.dinv[v] : 0.0f;
  float r = act ? a.r[v] : 0.0f, x = 0.0f, z = d * r;
  if (act) {
    __stcg(a.z + v, z);
    __stcg(a.p0 + v, 0.0f);
  }
  cluster_barrier();                         // every CTA has started: its memory may be written
  const int span = nvc + 2 * halo;
  double rz = 0.0;                           // warp 0
  int set = 0;
  float *pold = a.p0, *pnew = a.p1;
  // one reduction, then warp 0's thread 0 makes the step's coefficient
  auto meet = [&](double val, auto step) {
    const double t = cluster_sum(val, sw, slots[set]);
    set ^= 1;
    if (tid < 32) {
      const bool bad = dbits(t) <= 0 || is_nan(t);
      const float cf = step(t, bad);
      if (tid == 0) {
        s_stop = bad;
        s_coef = cf;
      }
    }
    __syncthreads();
  };
  meet(fx_prod(r, z), [&](double t, bool) {
    rz = t;
    return 0.0f;
  });
  for (int it = 0; it < a.iters && !s_stop; ++it) {
    const float beta = s_coef;
    for (int q = tid; q < span; q += kClusterThreads) {
      const int n = v0 - halo + q;
      s_p[q] = n >= 0 && n < nv ? fmaf(beta, __ldcg(pold + n), __ldcg(a.z + n)) : 0.0f;
    }
    __syncthreads();
    float w = 0.0f, p = 0.0f;
    if (act) {
      // neighbours outside the box have zero entries
      const float* sp = s_p + halo + tid;
      p = sp[0];
      __stcg(pnew + v, p);
#pragma unroll
      for (int o = 0; o < 27; ++o)
        w = fmaf(c[o], sp[o % 3 - 1 + a.nvx * ((o / 3) % 3 - 1 + a.nvy * (o / 9 - 1))], w);
    }
    meet(fx_prod(p, w),
         [&](double t, bool bad) { return bad ? 0.0f : ratio32(rz, t); });
    if (s_stop) break;
    const float alpha = s_coef;
    x = fmaf(alpha, p, x);
    r = fmaf(-alpha, w, r);
    z = d * r;
    if (it + 1 == a.iters) break;            // the last direction has been taken
    if (act) __stcg(a.z + v, z);
    meet(fx_prod(r, z), [&](double t, bool bad) {
      const float b = bad ? 0.0f : ratio32(t, rz);
      rz = t;
      return b;
    });
    float* t = pold;
    pold = pnew;
    pnew = t;
  }
  if (act) a.x[v] = x;
}

// L-vector of vertex function v (all elements), FP64
__global__ void k_vertex_field(int64_t nL, int P, int v, const double* __restrict__ xi,
                               double* __restrict__ out) {
  const int P3 = P * P * P;
  for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < nL;
       q += (int64_t)gridDim.x * blockDim.x) {
    const int lq = (int)(q % P3);
    const int i = lq % P, j = (lq / P) % P, k = lq / (P * P);
    const double fa = (v & 1) ? 0.5 * (1.0 + xi[i]) : 0.5 * (1.0 - xi[i]);
    const double fb = ((v >> 1) & 1) ? 0.5 * (1.0 + xi[j]) : 0.5 * (1.0 - xi[j]);
    const double fc = (v >> 2) ? 0.5 * (1.0 + xi[k]) : 0.5 * (1.0 - xi[k]);
    out[q] = fa * fb * fc;
  }
}

// K[e][pk(r, v)] = phi_r^T (H_e phi_v) for r <= v (one CTA per element)
__global__ void k_coarse_entries(int E, int P, int v, const double* __restrict__ hv,
                                 const double* __restrict__ xi, float* __restrict__ K,
                                 double* __restrict__ diag) {
  __shared__ double red[8][8];
  const int P3 = P * P * P;
  for (int e = blockIdx.x; e < E; e += gridDim.x) {
    double acc[8];
#pragma unroll
    for (int r = 0; r < 8; ++r) acc[r] = 0.0;
    for (int q = threadIdx.x; q < P3; q += blockDim.x) {
      const int i = q % P, j = (q / P) % P, k = q / (P * P);
      const double hq = hv[(size_t)e * P3 + q];
#pragma unroll
      for (int r = 0; r < 8; ++r) {
        const double fa = (r & 1) ? 0.5 * (1.0 + xi[i]) : 0.5 * (1.0 - xi[i]);
        const double fb = ((r >> 1) & 1) ? 0.5 * (1.0 + xi[j]) : 0.5 * (1.0 - xi[j]);
        const double fc = (r >> 2) ? 0.5 * (1.0 + xi[k]) : 0.5 * (1.0 - xi[k]);
        acc[r] += fa * fb * fc * hq;
      }
    }
#pragma unroll
    for (int r = 0; r < 8; ++r)
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) acc[r] += __shfl_down_sync(0xffffffffu, acc[r], o);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (lane == 0)
#pragma unroll
      for (int r = 0; r < 8; ++r) red[r][wid] = acc[r];
    __syncthreads();
    if (threadIdx.x < 8) {
      const int r = threadIdx.x;
      double t = 0.0;
      for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += red[r][w];
      if (r <= v) K[(size_t)e * 36 + pk(r, v)] = (float)t;
      if (r == v) diag[(size_t)e * 8 + v] = t;
    }
    __syncthreads();
  }
}

// cdinv[v] = mask_v / sum over elements of the vertex's diagonal entries
__global__ void k_coarse_dinv(int E, const double* __restrict__ diag, float* __restrict__ cdinv,
                              double* __restrict__ acc, int nelx, int nely, int nelz, int faces,
                              int phase) {
  const int nvx = nelx + 1, nvy = nely + 1, nvz = nelz + 1;
  if (phase == 0) {
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < E; e += gridDim.x * blockDim.x) {
      const int ex = e % nelx, ey = (e / nelx) % nely, ez = e / (nelx * nely);
      for (int v = 0; v < 8; ++v) {
        const int vi = (ex + (v & 1)) + nvx * ((ey + ((v >> 1) & 1)) + nvy * (ez + (v >> 2)));
        atomicAdd(acc + vi, diag[(size_t)e * 8 + v]);
      }
    }
  } else {
    const int nv = nvx * nvy * nvz;
    for (int vi = blockIdx.x * blockDim.x + threadIdx.x; vi < nv; vi += gridDim.x * blockDim.x) {
      const int x = vi % nvx, y = (vi / nvx) % nvy, z = vi / (nvx * nvy);
      const bool masked = ((faces & SEM_FACE_XMIN) && x == 0) || ((faces & SEM_FACE_XMAX) && x == nelx) ||
                          ((faces & SEM_FACE_YMIN) && y == 0) || ((faces & SEM_FACE_YMAX) && y == nely) ||
                          ((faces & SEM_FACE_ZMIN) && z == 0) || ((faces & SEM_FACE_ZMAX) && z == nelz);
      cdinv[vi] = masked || !(acc[vi] > 0.0) ? 0.0f : (float)(1.0 / acc[vi]);
    }
  }
}

// z_L = mask o (z_local[g(L)] + sum_v phi_v c_v) at every local point
template <int P>
__global__ void k_sw_combine(int64_t nL, const float* __restrict__ zg, const float* __restrict__ xc,
                             double* __restrict__ z, SwParams prm, int faces) {
  constexpr int N = P - 1, P3 = P * P * P;
  for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < nL;
       q += (int64_t)gridDim.x * blockDim.x) {
    const uint32_t e = (uint32_t)q / (uint32_t)P3;    // n_L < 2^31
    const int lq = (int)((uint32_t)q - e * (uint32_t)P3);
    const int i = lq % P, j = (lq / P) % P, k = lq / (P * P);
    const uint32_t re = prm.dnx.div(e);
    const int ex = (int)(e - re * (uint32_t)prm.nelx);
    const uint32_t ezu = prm.dny.div(re);
    const int ey = (int)(re - ezu * (uint32_t)prm.nely), ez = (int)ezu;
    const int ix = ex * N + i, iy = ey * N + j, iz = ez * N + k;
    const bool masked = ((faces & SEM_FACE_XMIN) && ix == 0) ||
                        ((faces & SEM_FACE_XMAX) && ix == prm.gx - 1) ||
                        ((faces & SEM_FACE_YMIN) && iy == 0) ||
                        ((faces & SEM_FACE_YMAX) && iy == prm.gy - 1) ||
                        ((faces & SEM_FACE_ZMIN) && iz == 0) ||
                        ((faces & SEM_FACE_ZMAX) && iz == N * prm.nelz);
    double v = 0.0;
    if (!masked) {
      v = (double)zg[(long long)ix + (long long)prm.gx * iy + prm.sk * iz];
      if (xc) {
        const int v0 = ex + (prm.nelx + 1) * (ey + (prm.nely + 1) * ez);
        const int sy = prm.nelx + 1, sz = (prm.nelx + 1) * (prm.nely + 1);
        const float fx0 = prm.phi[0][i], fx1 = prm.phi[1][i];
        const float fy0 = prm.phi[0][j], fy1 = prm.phi[1][j];
        const float fz0 = prm.phi[0][k], fz1 = prm.phi[1][k];
        const float c00 = fmaf(fx1, xc[v0 + 1], fx0 * xc[v0]);
        const float c10 = fmaf(fx1, xc[v0 + sy + 1], fx0 * xc[v0 + sy]);
        const float c01 = fmaf(fx1, xc[v0 + sz + 1], fx0 * xc[v0 + sz]);
        const float c11 = fmaf(fx1, xc[v0 + sz + sy + 1], fx0 * xc[v0 + sz + sy]);
        v += (double)fmaf(fz1, fmaf(fy1, c11, fy0 * c01), fz0 * fmaf(fy1, c10, fy0 * c00));
      }
    }
    z[q] = v;
  }
}

int ew_blocks(int64_t n) {
  return (int)std::max<int64_t>(1, std::min<int64_t>((n + 255) / 256, 8 * sem_num_sms()));
}

}  // namespace
}  // namespace sem

using namespace sem;

struct sem_schwarz {
  sem_handle* h = nullptr;
  int levels = 3, coarse_iters = 10;
  double h1 = 1.0, h2 = 0.0;
  int Pe = 0;
  SwParams prm{};
  DevBuf<float> tab;                       // FDM tables
  std::vector<float> tab_h;                // the same on the host
  int64_t nv = 0, nv4 = 0;                 // coarse vertices, padded
  DevBuf<float> K, cdinv, rc, xc, pc, wc;
  // the one-launch coarse CG (where the vertices fit the resident grid): A_0 as a
  // stencil, scaled residual, reduction partials, barrier
  DevBuf<float> stencil, zc;
  DevBuf<double> cpart;
  DevBuf<unsigned> cbar;
  bool cluster_ok = false;                 // in one cluster
  DevBuf<float> rg, zg;                    // fine global vectors
  DevBuf<CGState> st;
  DevBuf<double> partials;
};

namespace sem {
namespace {

template <int PE>
void launch_local(sem_schwarz* sw, const float* rg, float* zg, cudaStream_t s) {
  using L = SwLayout<PE>;
  SwConst<PE> k;
  for (int d = 0; d < 3; ++d)
    for (int a = 0; a < PE; ++a)
      for (int b = 0; b < PE; ++b)
        k.S[d][a * PE + b] = sw->tab_h[(d * 4) * L::TAB + PE * L::R + a * L::R + b];
  schwarz_local_kernel<PE><<<(unsigned)sw->h->E, SwCfg<PE>::THREADS, 0, s>>>(
      rg, zg, sw->rc.ptr, sw->tab.ptr, sw->prm, k);
  SEM_CHECK_LAUNCH();
}

void launch_local_any(sem_schwarz* sw, const float* rg, float* zg, cudaStream_t s) {
  switch (sw->Pe) {
    case 4: launch_local<4>(sw, rg, zg, s); break;
    case 5: launch_local<5>(sw, rg, zg, s); break;
    case 6: launch_local<6>(sw, rg, zg, s); break;
    case 7: launch_local<7>(sw, rg, zg, s); break;
    case 8: launch_local<8>(sw, rg, zg, s); break;
    case 9: launch_local<9>(sw, rg, zg, s); break;
    case 10: launch_local<10>(sw, rg, zg, s); break;
    case 11: launch_local<11>(sw, rg, zg, s); break;
    case 12: launch_local<12>(sw, rg, zg, s); break;
    case 13: launch_local<13>(sw, rg, zg, s); break;
    default: throw Error(SEM_ERR_ARG, "schwarz: unsupported order");
  }
}

// fills the host FDM tables in the layout of SwLayout<Pe>
void build_tables(sem_schwarz* sw, std::vector<float>& out) {
  const sem_handle* h = sw->h;
  const int N = h->N, Pe = N + 3, R = (Pe + 3) / 4 * 4, TAB = 2 * Pe * R + R;
  out.assign(12 * TAB, 0.0f);
  const int nel[3] = {h->nelx, h->nely, h->nelz};
  const int flo[3] = {SEM_FACE_XMIN, SEM_FACE_YMIN, SEM_FACE_ZMIN};
  const int fhi[3] = {SEM_FACE_XMAX, SEM_FACE_YMAX, SEM_FACE_ZMAX};
  for (int d = 0; d < 3; ++d) {
    const double L = h->len[d] / nel[d];
    for (int v = 0; v < 4; ++v) {
      const int bkind_lo = (h->faces & flo[d]) ? kDir : kFree;
      const int bkind_hi = (h->faces & fhi[d]) ? kDir : kFree;
      const int lo = (v & 1) ? bkind_lo : kNbr;
      const int hi = (v & 2) ? bkind_hi : kNbr;
      std::vector<double> A, B, V, lam;
      unsigned keep = 0;
      extended_1d(h, L, lo, hi, A, B, keep);
      sw->prm.keep[d][v] = keep;
      std::vector<double> C(Pe * Pe), bh(Pe);
      for (int a = 0; a < Pe; ++a) bh[a] = 1.0 / std::sqrt(B[a]);
      for (int a = 0; a < Pe; ++a)
        for (int b = 0; b < Pe; ++b) C[a * Pe + b] = bh[a] * A[a * Pe + b] * bh[b];
      for (int a = 0; a < Pe; ++a)           // symmetrise against rounding
        for (int b = a + 1; b < Pe; ++b) {
          const double m = 0.5 * (C[a * Pe + b] + C[b * Pe + a]);
          C[a * Pe + b] = C[b * Pe + a] = m;
        }
      jacobi_eigen(Pe, C, V, lam);
      float* t = out.data() + (d * 4 + v) * TAB;
      for (int a = 0; a < Pe; ++a)
        for (int ap = 0; ap < Pe; ++ap) {
          const double S = bh[a] * V[a * Pe + ap];     // S[a][a']
          t[ap * R + a] = (float)S;                    // ST[a'][a]
          t[Pe * R + a * R + ap] = (float)S;           // S[a][a']
        }
      for (int a = 0; a < Pe; ++a) t[2 * Pe * R + a] = (float)lam[a];
    }
  }
  auto lam0 = [&](int d, int a) { return out[d * 4 * TAB + 2 * Pe * R + a]; };
  const float h1 = sw->prm.h1, h2 = sw->prm.h2;
  for (int c = 0; c < Pe; ++c)
    for (int b = 0; b < Pe; ++b)
      for (int a = 0; a < Pe; ++a)
        out.push_back(std::fma(h1, lam0(0, a) + lam0(2, c) + lam0(1, b), h2));
}

int64_t coarse_cg_threads();
bool cluster_fits(const sem_schwarz* sw, cudaStream_t s);

// coarse element matrices from the FP64 element operator
void build_coarse(sem_schwarz* sw, cudaStream_t s) {
  sem_handle* h = sw->h;
  const int64_t nL = h->nL, E = h->E;
  sw->K.alloc((size_t)E * 36);
  DevBuf<double> phi, hphi, dg, acc, xi;
  phi.alloc(nL);
  hphi.alloc(nL);
  dg.alloc((size_t)E * 8);
  xi.alloc(h->P);
  xi.upload(h->xi.data(), h->P, s);
  for (int v = 0; v < 8; ++v) {
    k_vertex_field<<<ew_blocks(nL), 256, 0, s>>>(nL, h->P, v, xi.ptr, phi.ptr);
    SEM_CHECK_LAUNCH();
    launch_ax<double>(h, h->f64, phi.ptr, hphi.ptr, sw->h1, sw->h2, nullptr, nullptr, s);
    k_coarse_entries<<<(int)std::min<int64_t>(E, 8 * sem_num_sms()), 128, 0, s>>>(
        (int)E, h->P, v, hphi.ptr, xi.ptr, sw->K.ptr, dg.ptr);
    SEM_CHECK_LAUNCH();
  }
  acc.alloc(sw->nv);
  SEM_CUDA(cudaMemsetAsync(acc.ptr, 0, sw->nv * sizeof(double), s));
  SEM_CUDA(cudaMemsetAsync(sw->cdinv.ptr, 0, sw->nv4 * 4 * sizeof(float), s));
  k_coarse_dinv<<<ew_blocks(E), 256, 0, s>>>((int)E, dg.ptr, sw->cdinv.ptr, acc.ptr, h->nelx,
                                            h->nely, h->nelz, h->faces, 0);
  SEM_CHECK_LAUNCH();
  k_coarse_dinv<<<ew_blocks(sw->nv), 256, 0, s>>>((int)E, dg.ptr, sw->cdinv.ptr, acc.ptr,
                                                 h->nelx, h->nely, h->nelz, h->faces, 1);
  SEM_CHECK_LAUNCH();
  if (sw->nv <= coarse_cg_threads()) {
    sw->stencil.alloc((size_t)sw->nv * 27);
    sw->zc.alloc(sw->nv);
    sw->cpart.alloc(2 * 2 * kCoarseBlocks);
    sw->cbar.alloc(1);
    k_coarse_stencil<<<ew_blocks(sw->nv), 256, 0, s>>>(h->nelx, h->nely, h->nelz, sw->K.ptr,
                                                       sw->stencil.ptr, (int)sw->nv);
    SEM_CHECK_LAUNCH();
    sw->cluster_ok = cluster_fits(sw, s);
  }
  SEM_CUDA(cudaStreamSynchronize(s));      // the scratch buffers are freed on return
}

}  // namespace

sem_handle* schwarz_handle(const sem_schwarz* sw) { return sw->h; }

namespace {

// threads a grid of resident CTAs of the one-launch coarse CG has
int64_t coarse_cg_threads() {
  static const int occ = [] {
    const int smem = kCoarseBlocks * (int)sizeof(longlong2);
    int o = 0;
    SEM_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o, k_coarse_cg, kCoarseThreads, smem));
    return std::max(1, o);
  }();
  return (int64_t)std::min(kCoarseBlocks, occ * sem_num_sms()) * kCoarseThreads;
}

// the one-cluster form: vertices per CTA, neighbours kept on either side, launch
int cluster_share(const sem_schwarz* sw) {
  return (int)((sw->nv + kClusterCtas - 1) / kClusterCtas);
}
int cluster_halo(const sem_schwarz* sw) {
  const int nvx = sw->h->nelx + 1, nvy = sw->h->nely + 1;
  return nvx * nvy + nvx + 1;
}
cudaLaunchConfig_t cluster_config(const sem_schwarz* sw, cudaLaunchAttribute* at, cudaStream_t s) {
  at->id = cudaLaunchAttributeClusterDimension;
  at->val.clusterDim.x = kClusterCtas;
  at->val.clusterDim.y = 1;
  at->val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(kClusterCtas);
  cfg.blockDim = dim3(kClusterThreads);
  cfg.dynamicSmemBytes = (size_t)(cluster_share(sw) + 2 * cluster_halo(sw)) * sizeof(float);
  cfg.stream = s;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cfg;
}
// whether the vertices fit one cluster and the device can hold it
bool cluster_fits(const sem_schwarz* sw, cudaStream_t s) {
  if (cluster_share(sw) > kClusterThreads) return false;
  cudaLaunchAttribute at;
  const cudaLaunchConfig_t cfg = cluster_config(sw, &at, s);
  if (cfg.dynamicSmemBytes > 200 * 1024) return false;
  SEM_CUDA(cudaFuncSetAttribute(k_coarse_cluster, cudaFuncAttributeNonPortableClusterSizeAllowed,
                                1));
  SEM_CUDA(cudaFuncSetAttribute(k_coarse_cluster, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                200 * 1024));
  int n = 0;
  if (cudaOccupancyMaxActiveClusters(&n, k_coarse_cluster, &cfg) != cudaSuccess) {
    cudaGetLastError();                      // not a failure of the solve
    return false;
  }
  return n >= 1;
}

void launch_coarse_cg(sem_schwarz* sw, cudaStream_t s) {
  const sem_handle* h = sw->h;
  CoarseArgs a{};
  a.st = sw->stencil.ptr;
  a.dinv = sw->cdinv.ptr;
  a.r = sw->rc.ptr;
  a.x = sw->xc.ptr;
  a.p0 = sw->pc.ptr;
  a.p1 = sw->wc.ptr;
  a.z = sw->zc.ptr;
  a.partials = reinterpret_cast<longlong2*>(sw->cpart.ptr);
  a.bar = sw->cbar.ptr;
  a.err = h->dev_err.ptr;
  a.timeout_ns = kWaitTimeoutNs;
  a.nvx = h->nelx + 1;
  a.nvy = h->nely + 1;
  a.nvz = h->nelz + 1;
  a.iters = sw->coarse_iters;
  if (sw->cluster_ok) {
    cudaLaunchAttribute at;
    cudaLaunchConfig_t cfg = cluster_config(sw, &at, s);
    SEM_CUDA(cudaLaunchKernelEx(&cfg, k_coarse_cluster, a, cluster_share(sw), cluster_halo(sw)));
    return;
  }
  SEM_CUDA(cudaMemsetAsync(a.bar, 0, sizeof(unsigned), s));
  const int grid = (int)((sw->nv + kCoarseThreads - 1) / kCoarseThreads);
  void* args[] = {&a};
  SEM_CUDA(cudaLaunchCooperativeKernel(k_coarse_cg, dim3(grid), dim3(kCoarseThreads), args,
                                       grid * sizeof(longlong2), s));
}

}  // namespace

// the one-launch coarse CG of 2^3 vertices with a grid barrier that starts one
// arrival short, so that its first wait runs out; whether it gave up, recorded
// SEM_ERR_TIMEOUT in the handle's word and left NaN in its solution
bool selftest_coarse_timeout(const sem_handle* h, uint64_t timeout_ns, cudaStream_t s) {
  constexpr int nv = 8;
  DevBuf<float> f;                         // stencil, then dinv, r, x, p0, p1, z
  DevBuf<double> part;
  DevBuf<unsigned> bar;
  f.alloc(27 * nv + 6 * nv);
  part.alloc(4);
  bar.alloc(1);
  SEM_CUDA(cudaMemsetAsync(f.ptr, 0, f.n * sizeof(float), s));
  SEM_CUDA(cudaMemsetAsync(bar.ptr, 0xFF, sizeof(unsigned), s));
  CoarseArgs a{};
  float* v = f.ptr + 27 * nv;
  a.st = f.ptr;
  a.dinv = v;
  a.r = v + nv;
  a.x = v + 2 * nv;
  a.p0 = v + 3 * nv;
  a.p1 = v + 4 * nv;
  a.z = v + 5 * nv;
  a.partials = reinterpret_cast<longlong2*>(part.ptr);
  a.bar = bar.ptr;
  a.err = h->dev_err.ptr;
  a.timeout_ns = timeout_ns;
  a.nvx = a.nvy = a.nvz = 2;
  a.iters = 10;
  void* args[] = {&a};
  SEM_CUDA(cudaLaunchCooperativeKernel(k_coarse_cg, dim3(1), dim3(kCoarseThreads), args,
                                       sizeof(longlong2), s));
  float x[nv];
  int err = 0;
  SEM_CUDA(cudaMemcpyAsync(x, a.x, sizeof(x), cudaMemcpyDeviceToHost, s));
  SEM_CUDA(cudaMemcpyAsync(&err, h->dev_err.ptr, sizeof(int), cudaMemcpyDeviceToHost, s));
  SEM_CUDA(cudaStreamSynchronize(s));
  bool nan = true;
  for (float q : x) nan = nan && std::isnan(q);
  return err == (int)SEM_ERR_TIMEOUT && nan;
}

namespace {

// the local solves of rg added into zg (zeroed here), the coarse restriction
// and the coarse CG; returns the coarse solution or NULL (no coarse level)
const float* schwarz_levels(sem_schwarz* sw, const float* rg, float* zg, cudaStream_t s) {
  sem_handle* h = sw->h;
  SEM_CUDA(cudaMemsetAsync(zg, 0, h->nG * sizeof(float), s));
  const bool coarse = (sw->levels & SEM_SCHWARZ_COARSE) != 0;
  if (coarse) SEM_CUDA(cudaMemsetAsync(sw->rc.ptr, 0, sw->nv4 * 4 * sizeof(float), s));
  launch_local_any(sw, rg, zg, s);
  if (coarse && sw->stencil.ptr) {
    launch_coarse_cg(sw, s);
  } else if (coarse) {
    CGState* st = sw->st.ptr;
    vcg_init(sw->nv4, sw->rc.ptr, sw->cdinv.ptr, sw->pc.ptr, sw->xc.ptr, sw->wc.ptr, st,
             sw->partials.ptr, 0.0, sw->coarse_iters, s);
    const FastDiv dnx((uint32_t)h->nelx), dny((uint32_t)h->nely);
    for (int it = 0; it < sw->coarse_iters; ++it) {
      k_coarse_matvec<<<ew_blocks(h->E), 256, 0, s>>>((int)h->E, sw->K.ptr, sw->pc.ptr,
                                                      sw->wc.ptr, h->nelx, h->nely, dnx, dny);
      SEM_CHECK_LAUNCH();
      vcg_pw(sw->nv4, sw->pc.ptr, sw->wc.ptr, st, sw->partials.ptr, s);
      vcg_update(sw->nv4, sw->rc.ptr, sw->wc.ptr, sw->cdinv.ptr, st, nullptr, sw->partials.ptr, s);
      vcg_pupd(sw->nv4, sw->pc.ptr, sw->xc.ptr, sw->rc.ptr, sw->cdinv.ptr, st, s);
    }
  }
  return coarse ? sw->xc.ptr : nullptr;
}

// z_g = mask o (z_g + R_0^T c) at every global point.  A warp takes a row (iy,
// iz) of the lattice: its lanes blend the four coarse lines around the row with
// the y- and z-weights into shared memory, then the row's points take two
// entries each.  (A thread per point spent 33 us on 4.8 M points on index
// arithmetic and the eight coarse values; the bytes take 6 us.)
constexpr int kCombineWarps = 8;

__global__ void __launch_bounds__(32 * kCombineWarps, 6)
k_sw_combine_global(float* __restrict__ z, const float* __restrict__ xc,
                    const __grid_constant__ SwParams prm, int faces, int rows, int gy, FastDiv dgy,
                    FastDiv dN, int use_line) {
  extern __shared__ float s_line[];
  constexpr int Q = 4;                     // points a lane has on their way
  const int N = prm.N, lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nvx = prm.nelx + 1;
  float* line = s_line + warp * nvx;
  __shared__ float s_phi[2][kMaxP];
  if (threadIdx.x < 2 * kMaxP)
    s_phi[threadIdx.x / kMaxP][threadIdx.x % kMaxP] =
        prm.phi[threadIdx.x / kMaxP][threadIdx.x % kMaxP];
  __syncthreads();
  const int row = blockIdx.x * kCombineWarps + warp;
  if (row >= rows) return;
  const int iz = (int)dgy.div((uint32_t)row), iy = row - iz * gy;
  float* zr = z + (long long)row * prm.gx;
  const bool masked = ((faces & SEM_FACE_YMIN) && iy == 0) ||
                      ((faces & SEM_FACE_YMAX) && iy == N * prm.nely) ||
                      ((faces & SEM_FACE_ZMIN) && iz == 0) ||
                      ((faces & SEM_FACE_ZMAX) && iz == N * prm.nelz);
  if (masked) {
    for (int ix = lane; ix < prm.gx; ix += 32) zr[ix] = 0.0f;
    return;
  }
  float t[Q];
#pragma unroll
  for (int q = 0; q < Q; ++q) t[q] = lane + 32 * q < prm.gx ? zr[lane + 32 * q] : 0.0f;
  const int ey = min((int)dN.div((uint32_t)iy), prm.nely - 1);
  const int ez = min((int)dN.div((uint32_t)iz), prm.nelz - 1);
  const int sy = nvx, sz = nvx * (prm.nely + 1);
  const float* c0 = xc + (ey * sy + ez * sz);
  const float fy0 = s_phi[0][iy - ey * N], fy1 = s_phi[1][iy - ey * N];
  const float fz0 = s_phi[0][iz - ez * N], fz1 = s_phi[1][iz - ez * N];
  auto blend = [&](int v) {
    return fmaf(fz1, fmaf(fy1, c0[v + sz + sy], fy0 * c0[v + sz]),
                fz0 * fmaf(fy1, c0[v + sy], fy0 * c0[v]));
  };
  if (xc && use_line) {
    for (int v = lane; v < nvx; v += 32) line[v] = blend(v);
    __syncwarp();
  }
  const int last = prm.gx - 1;
  const bool m0 = (faces & SEM_FACE_XMIN) != 0, m1 = (faces & SEM_FACE_XMAX) != 0;
  for (int i0 = lane; i0 < prm.gx; i0 += 32 * Q) {
    if (i0 != lane)
#pragma unroll
      for (int q = 0; q < Q; ++q) t[q] = i0 + 32 * q < prm.gx ? zr[i0 + 32 * q] : 0.0f;
#pragma unroll
    for (int q = 0; q < Q; ++q) {
      const int ix = i0 + 32 * q;
      if (ix >= prm.gx) break;
      float v = t[q];
      if (xc) {
        const int ex = min((int)dN.div((uint32_t)ix), prm.nelx - 1), i = ix - ex * N;
        const float c1 = use_line ? line[ex + 1] : blend(ex + 1), cl = use_line ? line[ex] : blend(ex);
        v += fmaf(s_phi[1][i], c1, s_phi[0][i] * cl);
      }
      zr[ix] = (m0 && ix == 0) || (m1 && ix == last) ? 0.0f : v;
    }
  }
}

}  // namespace

void schwarz_apply_global(sem_schwarz* sw, const float* r_g, float* z_g, cudaStream_t s) {
  sem_handle* h = sw->h;
  const float* xcp = schwarz_levels(sw, r_g, z_g, s);
  const int gy = h->N * h->nely + 1, rows = gy * (h->N * h->nelz + 1);
  const int blocks = (rows + kCombineWarps - 1) / kCombineWarps;
  size_t smem = (size_t)kCombineWarps * (h->nelx + 1) * sizeof(float);
  const int use_line = smem <= 32 * 1024 ? 1 : 0;      // over 1000 elements along x: no lines
  if (!use_line) smem = 0;
  k_sw_combine_global<<<blocks, 32 * kCombineWarps, smem, s>>>(
      z_g, xcp, sw->prm, h->faces, rows, gy, FastDiv((uint32_t)gy), FastDiv((uint32_t)h->N),
      use_line);
  SEM_CHECK_LAUNCH();
}

void schwarz_apply(sem_schwarz* sw, const double* r, double* z, cudaStream_t s) {
  sem_handle* h = sw->h;
  to_global<double>(h, r, sw->rg.ptr, s);
  const float* xcp = schwarz_levels(sw, sw->rg.ptr, sw->zg.ptr, s);
  const int cg = ew_blocks(h->nL);
  switch (h->P) {
    case 3: k_sw_combine<3><<<cg, 256, 0, s>>>(h->nL, sw->zg.ptr, xcp, z, sw->prm, h->faces); break;
    case 4: k_sw_combine<4><<<cg, 256, 0, s>>>(h->nL, sw->zg.ptr, xcp, z, sw->prm, h->faces); break;
    case 5: k_sw_combine<5><<<cg, 256, 0, s>>>(h->nL, sw->zg.ptr, xcp, z, sw->prm, h->faces); break;
    case 6: k_sw_combine<6><<<cg, 256, 0, s>>>(h->nL, sw->zg.ptr, xcp, z, sw->prm, h->faces); break;
    case 7: k_sw_combine<7><<<cg, 256, 0, s>>>(h->nL, sw->zg.ptr, xcp, z, sw->prm, h->faces); break;
    case 8: k_sw_combine<8><<<cg, 256, 0, s>>>(h->nL, sw->zg.ptr, xcp, z, sw->prm, h->faces); break;
    case 9: k_sw_combine<9><<<cg, 256, 0, s>>>(h->nL, sw->zg.ptr, xcp, z, sw->prm, h->faces); break;
    case 10: k_sw_combine<10><<<cg, 256, 0, s>>>(h->nL, sw->zg.ptr, xcp, z, sw->prm, h->faces); break;
    case 11: k_sw_combine<11><<<cg, 256, 0, s>>>(h->nL, sw->zg.ptr, xcp, z, sw->prm, h->faces); break;
    default: throw Error(SEM_ERR_ARG, "schwarz: unsupported order");
  }
  SEM_CHECK_LAUNCH();
}

}  // namespace sem

extern "C" sem_status sem_schwarz_create(sem_handle* h, double h1, double h2, int levels,
                                         int coarse_iters, void* stream, sem_schwarz** out) {
  return guarded("sem_schwarz_create", [&] {
    SEM_REQUIRE(h && out, "sem_schwarz_create: null argument");
    *out = nullptr;
    SEM_REQUIRE(levels >= 1 && levels <= 3, "sem_schwarz_create: levels must be 1, 2 or 3");
    SEM_REQUIRE(coarse_iters >= 0 && coarse_iters <= 1000,
                "sem_schwarz_create: coarse_iters must be in [0, 1000]");
    SEM_REQUIRE(h1 > 0.0 && h2 >= 0.0, "sem_schwarz_create: needs h1 > 0 and h2 >= 0");
    SEM_REQUIRE(h->N >= 2, "sem_schwarz_create: needs N >= 2 (the point a subdomain takes from "
                           "a neighbour must lie inside it)");
    cudaStream_t s = (cudaStream_t)stream;
    std::unique_ptr<sem_schwarz> sw(new sem_schwarz());
    sw->h = h;
    sw->levels = levels;
    sw->coarse_iters = coarse_iters;
    sw->h1 = h1;
    sw->h2 = h2;
    sw->Pe = h->N + 3;
    SwParams& p = sw->prm;
    p.N = h->N;
    p.nelx = h->nelx; p.nely = h->nely; p.nelz = h->nelz;
    p.gx = h->N * h->nelx + 1;
    p.gy = h->N * h->nely + 1;
    p.sk = (long long)p.gx * p.gy;
    p.dnx = FastDiv((uint32_t)h->nelx);
    p.dny = FastDiv((uint32_t)h->nely);
    p.h1 = (float)h1;
    p.h2 = (float)h2;
    p.do_local = (levels & SEM_SCHWARZ_LOCAL) ? 1 : 0;
    p.do_coarse = (levels & SEM_SCHWARZ_COARSE) ? 1 : 0;
    for (int i = 0; i < h->P; ++i) {
      p.phi[0][i] = (float)(0.5 * (1.0 - h->xi[i]));
      p.phi[1][i] = (float)(0.5 * (1.0 + h->xi[i]));
    }
    build_tables(sw.get(), sw->tab_h);
    sw->tab.alloc(sw->tab_h.size());
    sw->tab.upload(sw->tab_h.data(), sw->tab_h.size(), s);
    sw->rg.alloc(h->nG);
    sw->zg.alloc(h->nG);
    sw->nv = (int64_t)(h->nelx + 1) * (h->nely + 1) * (h->nelz + 1);
    sw->nv4 = (sw->nv + 3) / 4;
    for (DevBuf<float>* b : {&sw->cdinv, &sw->rc, &sw->xc, &sw->pc, &sw->wc}) {
      b->alloc(sw->nv4 * 4);
      SEM_CUDA(cudaMemsetAsync(b->ptr, 0, sw->nv4 * 4 * sizeof(float), s));
    }
    sw->st.alloc(1);
    SEM_CUDA(cudaMemsetAsync(sw->st.ptr, 0, sizeof(CGState), s));
    sw->partials.alloc(2 * kRedBlocks);
    if (levels & SEM_SCHWARZ_COARSE) build_coarse(sw.get(), s);
    SEM_CUDA(cudaStreamSynchronize(s));
    *out = sw.release();
  });
}

extern "C" sem_status sem_schwarz_apply(sem_schwarz* sw, const double* r_L, double* z_L,
                                        void* stream) {
  return guarded("sem_schwarz_apply", [&] {
    SEM_REQUIRE(sw && r_L && z_L, "sem_schwarz_apply: null argument");
    SEM_REQUIRE(r_L != z_L, "sem_schwarz_apply: r and z must not alias");
    schwarz_apply(sw, r_L, z_L, (cudaStream_t)stream);
  });
}

extern "C" sem_status sem_schwarz_destroy(sem_schwarz* sw) {
  return guarded("sem_schwarz_destroy", [&] {
    if (sw) cudaDeviceSynchronize();
    delete sw;
  });
}
