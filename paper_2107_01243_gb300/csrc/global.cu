// The FP32 operator on global (unique-dof) vectors, w_g = mask Q^T (h1 A_L +
// h2 B_L) Q u_g (arXiv 2107.01243 §2, Eq. 9-10, with the local-to-global map
// Q of Eq. 10 applied inside the element kernel), for the FP32 inner solves
// of the mixed-precision solver, and the conversions between L-vectors and
// global vectors.
//
// On the box the global numbering is the lattice g = ix + gx (iy + gy iz), so
// an element gathers its P^3 values as P^2 rows of P consecutive floats of
// the lattice (the faces it shares are read again, from L2, by its
// neighbours), and assembles its output directly: points inside the element
// belong to it alone and are stored, points on its faces are added with
// atomics (reductions in L2), Dirichlet points are skipped.  Global vectors
// hold about (N/(N+1))^3 of the local points (0.67 at N = 7), so each CG
// vector pass moves a third fewer bytes, and no gather-scatter pass is left.
// The order of the atomic additions varies, so FP32 results may differ in
// the last bits from run to run; the FP64 refinement around the inner solve
// is unaffected.
#include <cmath>

#include "sem_internal.cuh"
#include "tma.cuh"
#include "ax_line.cuh"
#include "fixsum.cuh"
#include "reduce.cuh"
#include "cg_state.cuh"

namespace sem {

struct GBox {
  int nelx, nely, nelz, faces;
  int gx;             // lattice extent in x
  long long sk;       // lattice stride in z: gx gy
  FastDiv dnx, dny;   // division by nelx, nely
};

// box position of element e and the lattice index of its point (0, 0, 0)
__device__ __forceinline__ long long elem_origin(int e, const GBox& b, int N, int& ex, int& ey,
                                                 int& ez) {
  const uint32_t r = b.dnx.div((uint32_t)e);
  ex = e - (int)r * b.nelx;
  const uint32_t q = b.dny.div(r);
  ey = (int)(r - q * (uint32_t)b.nely);
  ez = (int)q;
  return (long long)(ex * N) + (long long)b.gx * (ey * N) + b.sk * (long long)(ez * N);
}

// Dirichlet face bits of element (ex, ey, ez) in the point-flag layout below
__device__ __forceinline__ unsigned dirichlet_bits(const GBox& b, int ex, int ey, int ez) {
  if (!b.faces) return 0u;
  return ((b.faces & SEM_FACE_XMIN) && ex == 0 ? 4u : 0u) |
         ((b.faces & SEM_FACE_XMAX) && ex == b.nelx - 1 ? 8u : 0u) |
         ((b.faces & SEM_FACE_YMIN) && ey == 0 ? 16u : 0u) |
         ((b.faces & SEM_FACE_YMAX) && ey == b.nely - 1 ? 32u : 0u) |
         ((b.faces & SEM_FACE_ZMIN) && ez == 0 ? 64u : 0u) |
         ((b.faces & SEM_FACE_ZMAX) && ez == b.nelz - 1 ? 128u : 0u);
}

// A CTA takes K consecutive elements (ax_line.cuh): every thread
// gathers its own k-column of u from the lattice (rows of P consecutive floats;
// what neighbours share comes from L2) and scatters its column of outputs.
// With the clearing of w, on 17 M points: N = 3 102 us, N = 5 115, N = 7 101, N = 9
// 135 (Poisson; with a mass term 112, 131, 106, 138).  The kernel it took the
// place of staged G by bulk copies and read a row and a column of shared memory
// for every point: 149, 146, 113, 150 (154, 150, 128, 153).  w
// must hold zeros at every unmasked point on element faces.
// PW: <p, H p> from the local products, p = u (the sum over local
// points of u_L (H_L u_L), equal to the global product because u is zero on
// Dirichlet points), every warp's sum added to one of kPwSlots accumulators (in
// no fixed order, as the face sums of w).
// No loop over elements: with one the compiler keeps D in registers.
// The operator alone at N = 9 fetches three components of G ahead instead of six,
// so that six CTAs fit an SM instead of four: 138 us (h2 = 0: 135).  With the
// Kahan sum (PW, and batch_glob.cuh) the registers do not allow it: 16 problems
// with 17,000 elements of N = 9 187 against 169 us.
// FEW: at most a CTA an SM, where a late load's latency counts and registers do
// not: all six components ahead (N = 9, 8 to 64 elements, cold caches: 11.1 to 12.5
// against 12.3 to 13.3 us).
template <int P, bool PW, bool FEW>
struct GlobCfg : LineCfg<P, float, kGlobThreads> {
  static constexpr bool LEAN = P >= 10 && !PW && !FEW;
  static constexpr int PREG = LEAN ? 3 : 6;
  static constexpr int CTAS = LEAN ? 6 : LineCfg<P, float, kGlobThreads>::MINB;
};

template <int P, bool PW, bool FEW>
__global__ void __launch_bounds__(GlobCfg<P, PW, FEW>::THREADS, GlobCfg<P, PW, FEW>::CTAS)
ax_glob_kernel(const float* __restrict__ u, float* __restrict__ w, const float* __restrict__ G,
               const float* __restrict__ B, float h1, float h2,
               const __grid_constant__ DMat<P, float> D, int E, GBox bx,
               const CGState* __restrict__ st, double* __restrict__ slots) {
  using C = GlobCfg<P, PW, FEW>;
  constexpr int P3 = C::P3, K = C::K, N = P - 1;
  if (st && st->done) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  LineThread<P, float, kGlobThreads> t;
  t.init(smem_raw);
  const int toff = t.i + bx.gx * t.j, sk = (int)bx.sk;      // n_G < 2^31
  const bool fij = t.i == 0 || t.i == N || t.j == 0 || t.j == N;
  const unsigned pij = (t.i == 0 ? 4u : 0u) | (t.i == N ? 8u : 0u) | (t.j == 0 ? 16u : 0u) |
                       (t.j == N ? 32u : 0u);
  const int e = blockIdx.x * K + t.el;
  const bool act = t.el < K && e < E;
  int ex, ey, ez;
  const int org = (int)elem_origin(act ? e : 0, bx, N, ex, ey, ez) + toff;
  float uc[P], out[P];
  if (act) {
#pragma unroll
    for (int k = 0; k < P; ++k) uc[k] = __ldg(u + (org + sk * k));
  }
  const size_t base = (size_t)(act ? e : 0) * P3 + t.lam;
  line_element<C::PREG>(t, act, D, uc, G + (size_t)(act ? e : 0) * 6 * P3 + t.lam,
                        B + base, (const float*)nullptr, h1, h2, out);
  float pw = 0.0f, pw_c = 0.0f;            // Kahan-compensated <p, H p>
  if (act) {
    int dst0 = org;                        // the column's addresses are made anew:
    asm volatile("" : "+r"(dst0));         // kept since the gather they would spill
    const unsigned fl = dirichlet_bits(bx, ex, ey, ez);
#pragma unroll
    for (int k = 0; k < P; ++k) {
      if (PW) {
        const float y = __fsub_rn(__fmul_rn(uc[k], out[k]), pw_c);
        const float tt = __fadd_rn(pw, y);
        pw_c = __fsub_rn(__fsub_rn(tt, pw), y);
        pw = tt;
      }
      const unsigned pf = pij | (k == 0 ? 64u : 0u) | (k == N ? 128u : 0u);
      if (pf & fl) continue;               // Dirichlet point: stays zero
      float* dst = w + (dst0 + sk * k);
      if (fij || k == 0 || k == N)
        red_add(dst, out[k]);              // shared with neighbours
      else
        *dst = out[k];                     // interior: this element's alone
    }
  }
  if constexpr (PW) {
    constexpr int NW = C::THREADS / 32;
    const FxVal f = fx_warp_sum(pw, pw_c);
    if ((threadIdx.x & 31) == 0)
      atomicAdd(slots + (blockIdx.x * NW + (threadIdx.x >> 5)) % kPwSlots,
                fx_round(f.m >> 32, (long long)(unsigned)f.m, f.e));
  }
}

static GBox make_gbox(const sem_handle* h) {
  GBox b;
  b.nelx = h->nelx;
  b.nely = h->nely;
  b.nelz = h->nelz;
  b.faces = h->faces;
  b.gx = h->N * h->nelx + 1;
  b.sk = (long long)b.gx * (h->N * h->nely + 1);
  b.dnx = FastDiv((uint32_t)h->nelx);
  b.dny = FastDiv((uint32_t)h->nely);
  return b;
}

double* pw_slots(const sem_handle* h) {
  return h->partials.ptr + 6 * kRedBlocks + kFusedPartials;
}

template <int P, bool PW, bool FEW>
static void configure_glob() {
  static const bool done = [] {
    SEM_CUDA(cudaFuncSetAttribute(ax_glob_kernel<P, PW, FEW>,
                                  cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)GlobCfg<P, PW, FEW>::SMEM));
    return true;
  }();
  (void)done;
}

template <int P, bool PW, bool FEW>
static void launch_glob_p(const sem_handle* h, const float* u, float* w, float h1, float h2,
                          const CGState* st, cudaStream_t s) {
  using C = GlobCfg<P, PW, FEW>;
  auto kern = ax_glob_kernel<P, PW, FEW>;
  configure_glob<P, PW, FEW>();
  DMat<P, float> D;
  for (int a = 0; a < P * P; ++a) D.d[a] = (float)h->Dh[a];
  const int E = (int)h->E;
  kern<<<(E + C::K - 1) / C::K, C::THREADS, C::SMEM, s>>>(u, w, h->f32.G.ptr, h->f32.B.ptr, h1, h2,
                                                          D, E, make_gbox(h), st, pw_slots(h));
  SEM_CHECK_LAUNCH();
}

bool glob_supported(const sem_handle* h) {
  const int P = h->P;
  return h->f32.G.ptr && (P == 2 || P == 4 || P == 6 || P == 8 || P == 10) && h->E > 0 &&
         h->nL < (1LL << 31);
}

int64_t glob_padded(const sem_handle* h) { return (h->nG + 3) / 4 * 4; }

template <int P>
static void launch_glob_any(const sem_handle* h, const float* u, float* w, float h1, float h2,
                            const CGState* st, bool pw, cudaStream_t s) {
  if (pw) return launch_glob_p<P, true, false>(h, u, w, h1, h2, st, s);
  if constexpr (P == 10)
    if (h->E <= sem_num_sms()) return launch_glob_p<P, false, true>(h, u, w, h1, h2, st, s);
  launch_glob_p<P, false, false>(h, u, w, h1, h2, st, s);
}

template <int P>
static void configure_glob_any() {
  configure_glob<P, true, false>();
  configure_glob<P, false, false>();
  if constexpr (P == 10) configure_glob<P, false, true>();
}

// once-per-process kernel attributes, set by sem_setup outside any stream capture
void glob_kernel_prepare(const sem_handle* h) {
  if (!h->f32.G.ptr) return;
  switch (h->P) {
    case 2: return configure_glob_any<2>();
    case 4: return configure_glob_any<4>();
    case 6: return configure_glob_any<6>();
    case 8: return configure_glob_any<8>();
    case 10: return configure_glob_any<10>();
  }
}

void launch_apply_global(const sem_handle* h, const float* u, float* w, float h1, float h2,
                         const CGState* st, bool pw, cudaStream_t s) {
  switch (h->P) {
    case 2: launch_glob_any<2>(h, u, w, h1, h2, st, pw, s); break;
    case 4: launch_glob_any<4>(h, u, w, h1, h2, st, pw, s); break;
    case 6: launch_glob_any<6>(h, u, w, h1, h2, st, pw, s); break;
    case 8: launch_glob_any<8>(h, u, w, h1, h2, st, pw, s); break;
    case 10: launch_glob_any<10>(h, u, w, h1, h2, st, pw, s); break;
    default: throw Error(SEM_ERR_ARG, "apply_global: unsupported order");
  }
}

// ---------------------------------------------------------------- conversions
// Thread per global point g = ix + gx (iy + gy iz): reads the copy of g in
// element (ex, ey, ez) = (min(ix / N, nelx - 1), likewise y, z); the input is
// continuous, so every copy holds the same value.
template <class Tin>
__global__ void k_to_global(int64_t nG, const Tin* __restrict__ in, float* __restrict__ out,
                            int N, int P, int nelx, int nely, int nelz, FastDiv dgx, FastDiv dgy,
                            FastDiv dN, double scale) {
  const long long P3 = (long long)P * P * P;
  for (int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; g < nG;
       g += (int64_t)gridDim.x * blockDim.x) {
    const uint32_t r = dgx.div((uint32_t)g);
    const int ix = (int)((uint32_t)g - r * dgx.d);
    const uint32_t izu = dgy.div(r);
    const int iy = (int)(r - izu * dgy.d), iz = (int)izu;
    const int ex = min((int)dN.div((uint32_t)ix), nelx - 1);
    const int ey = min((int)dN.div((uint32_t)iy), nely - 1);
    const int ez = min((int)dN.div((uint32_t)iz), nelz - 1);
    const int i = ix - ex * N, j = iy - ey * N, k = iz - ez * N;
    const long long e = ex + (long long)nelx * (ey + (long long)nely * ez);
    out[g] = (float)((double)in[e * P3 + ((long long)k * P + j) * P + i] * scale);
  }
}

// x_L += d_g[g(L)] at every local point
__global__ void k_add_from_global(int64_t nL, double* __restrict__ x, const float* __restrict__ d,
                                  int N, int P, int nelx, int nely, int gx, int gy, FastDiv dP3,
                                  FastDiv dP, FastDiv dnx, FastDiv dny, double scale) {
  for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < nL;
       q += (int64_t)gridDim.x * blockDim.x) {
    const uint32_t qq = (uint32_t)q;
    const uint32_t e = dP3.div(qq);
    const uint32_t lq = qq - e * dP3.d;
    const uint32_t r1 = dP.div(lq);
    const uint32_t i = lq - r1 * (uint32_t)P;
    const uint32_t k = dP.div(r1);
    const uint32_t j = r1 - k * (uint32_t)P;
    const uint32_t re = dnx.div(e);
    const uint32_t ex = e - re * (uint32_t)nelx;
    const uint32_t ez = dny.div(re);
    const uint32_t ey = re - ez * (uint32_t)nely;
    const long long g = (long long)(ex * N + i) +
                        (long long)gx * ((long long)(ey * N + j) + (long long)gy * (ez * N + k));
    x[q] += (double)d[g] * scale;
  }
}

static int conv_grid(int64_t n) {
  return (int)std::max<int64_t>(1, std::min<int64_t>((n + 255) / 256, 8 * sem_num_sms()));
}

template <class Tin>
void to_global(const sem_handle* h, const Tin* in, float* out, cudaStream_t s, double scale) {
  const int N = h->N;
  k_to_global<Tin><<<conv_grid(h->nG), 256, 0, s>>>(
      h->nG, in, out, N, h->P, h->nelx, h->nely, h->nelz, FastDiv((uint32_t)(N * h->nelx + 1)),
      FastDiv((uint32_t)(N * h->nely + 1)), FastDiv((uint32_t)(N > 0 ? N : 1)), scale);
  SEM_CHECK_LAUNCH();
}
template void to_global<float>(const sem_handle*, const float*, float*, cudaStream_t, double);
template void to_global<double>(const sem_handle*, const double*, float*, cudaStream_t, double);

void add_from_global(const sem_handle* h, double* x, const float* d, cudaStream_t s,
                     double scale) {
  k_add_from_global<<<conv_grid(h->nL), 256, 0, s>>>(
      h->nL, x, d, h->N, h->P, h->nelx, h->nely, h->N * h->nelx + 1, h->N * h->nely + 1,
      FastDiv((uint32_t)h->P3), FastDiv((uint32_t)h->P), FastDiv((uint32_t)h->nelx),
      FastDiv((uint32_t)h->nely), scale);
  SEM_CHECK_LAUNCH();
}

}  // namespace sem

using namespace sem;

extern "C" sem_status sem_apply_global(sem_handle* h, const void* u_g, void* w_g, double h1,
                                       double h2, int dtype, void* stream) {
  return guarded("sem_apply_global", [&] {
    SEM_REQUIRE(h && u_g && w_g, "sem_apply_global: null argument");
    SEM_REQUIRE(u_g != w_g, "sem_apply_global: u and w must not alias");
    SEM_REQUIRE(dtype == SEM_F32, "sem_apply_global: FP32 only");
    SEM_REQUIRE(glob_supported(h), "sem_apply_global: needs FP32 geometry, an odd order N "
                                   "and fewer than 2^31 local points");
    const cudaStream_t s = (cudaStream_t)stream;
    SEM_CUDA(cudaMemsetAsync(w_g, 0, h->nG * sizeof(float), s));
    launch_apply_global(h, (const float*)u_g, (float*)w_g, (float)h1, (float)h2, nullptr, false,
                        s);
  });
}

extern "C" sem_status sem_to_global(sem_handle* h, const void* in_L, void* out_g, int dtype,
                                    void* stream) {
  return guarded("sem_to_global", [&] {
    SEM_REQUIRE(h && in_L && out_g, "sem_to_global: null argument");
    SEM_REQUIRE(dtype == SEM_F32 || dtype == SEM_F64, "sem_to_global: dtype");
    SEM_REQUIRE(h->nL < (1LL << 31), "sem_to_global: needs fewer than 2^31 local points");
    if (dtype == SEM_F32)
      to_global<float>(h, (const float*)in_L, (float*)out_g, (cudaStream_t)stream);
    else
      to_global<double>(h, (const double*)in_L, (float*)out_g, (cudaStream_t)stream);
  });
}
