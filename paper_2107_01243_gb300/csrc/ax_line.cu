// Element operator w_e = (h1 D^T G_e D + h2 B_e) u_e (arXiv 2107.01243 §2,
// Eq. 9) from plain coalesced loads at any alignment: the FP32 kernel of every P
// (elements of odd P are no whole number of 16 bytes, so that bulk copies cannot
// fetch them) and the IEEE FP64 kernel of large meshes at P = 8 and 10.
//
// A CTA takes K consecutive elements, K chosen so that K P^2 threads fill whole
// warps (P = 7: five elements, 245 of 256 lanes).  Thread (i, j) of an element
// owns the k-column: u and the t-direction stay in registers.  The r- and
// s-derivatives run as line tasks through shared memory: a thread reads one
// line of P values and makes its P outputs, so a point costs 15 shared-memory
// accesses in all instead of the 6 P of a column kernel that reads a row, a
// column and D's entries for every point (that kernel spent twice the HBM time
// of its bytes on shared memory at P = 7).  FP32: D's entries are constant-bank
// operands and G is on its way to registers before the forward lines run.
// FP64: GB300's FP64 pipe is the bound, so the lines use the even-odd split
// (eo_tile.cuh), which saves a quarter of the operations.
//
// FUSE: the output of the assembled operator (apply.cu): masked points are
// zero, and the x-pairs between the CTA's elements are summed through shared
// memory.
#include <type_traits>

#include "sem_internal.cuh"
#include "ax_tile.cuh"
#include "ax_line.cuh"

namespace sem {

// FIELD (FP32; FP64 looks at h1f): a per-point h1 is given, its column fetched with G
// and two CTAs made to fit an SM (one takes up to 38% longer at N = 9, 10)
template <int P, class T, bool FUSE, bool FIELD>
__global__ void __launch_bounds__(LineCfg<P, T>::THREADS,
                                  sizeof(T) == 4 && FIELD ? 2 : LineCfg<P, T>::MINB)
ax_line_kernel(const T* __restrict__ u, T* __restrict__ w, const T* __restrict__ G,
               const T* __restrict__ B, const T* __restrict__ h1f, T h1, T h2,
               const __grid_constant__ DMat<P, T> D, const T* __restrict__ tabg, int E, FuseBox fb,
               const CGState* __restrict__ st) {
  using C = LineCfg<P, T>;
  constexpr int P2 = C::P2, P3 = C::P3, K = C::K, N = P - 1;
  if (st && st->done) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  LineThread<P, T> t;
  t.init(smem_raw);
  if constexpr (C::TS > 0)
    for (int q = threadIdx.x; q < C::TS; q += C::THREADS) t.tab[q] = tabg[q];
  const int e = blockIdx.x * K + t.el;
  const bool act = t.el < K && e < E;
  const size_t base = (size_t)(act ? e : 0) * P3 + t.lam;
  T uc[P], out[P];
  if (act) {
#pragma unroll
    for (int k = 0; k < P; ++k) uc[k] = u[base + k * P2];
  }
  line_element<6, FIELD>(t, act, D, uc, G + (size_t)(act ? e : 0) * 6 * P3 + t.lam, B + base,
                         h1f ? h1f + base : nullptr, h1, h2, out);
  if constexpr (FUSE) {
    // masked points, then the x-pairs of neighbours in this CTA: the faces
    // i = 0 and i = N of every element go through U
    const int i = t.i, j = t.j;
    int ex = 0;
    if (act) {
      const int re = e / fb.nelx, ez = re / fb.nely, ey = re - ez * fb.nely, f = fb.faces;
      ex = e - re * fb.nelx;
      const bool mij = ((f & SEM_FACE_XMIN) && ex == 0 && i == 0) ||
                       ((f & SEM_FACE_XMAX) && ex == fb.nelx - 1 && i == N) ||
                       ((f & SEM_FACE_YMIN) && ey == 0 && j == 0) ||
                       ((f & SEM_FACE_YMAX) && ey == fb.nely - 1 && j == N);
#pragma unroll
      for (int k = 0; k < P; ++k)
        if (mij || (k == 0 && (f & SEM_FACE_ZMIN) && ez == 0) ||
            (k == N && (f & SEM_FACE_ZMAX) && ez == fb.nelz - 1))
          out[k] = T(0);
      if (i == 0 || i == N) {
#pragma unroll
        for (int k = 0; k < P; ++k) t.U[(i ? P2 : 0) + k * P + j] = out[k];
      }
    }
    __syncthreads();
    if (act) {
      const T* nb = nullptr;                 // the neighbour's copies of this column
      if (i == 0 && ex > 0 && t.el > 0) nb = t.U - C::VOL + P2 + j;
      if (i == N && ex < fb.nelx - 1 && t.el < K - 1) nb = t.U + C::VOL + j;
      if (nb) {
#pragma unroll
        for (int k = 0; k < P; ++k) out[k] += nb[k * P];
      }
    }
  }
  if (act) {
#pragma unroll
    for (int k = 0; k < P; ++k) w[base + k * P2] = out[k];
  }
}

// once-per-process kernel attributes, set by sem_setup outside any stream capture
template <int P, class T>
static void configure_line() {
  using C = LineCfg<P, T>;
  static const bool done = [] {
    constexpr bool F = sizeof(T) == 4;
    for (auto k : {ax_line_kernel<P, T, true, false>, ax_line_kernel<P, T, false, false>,
                   ax_line_kernel<P, T, true, F>, ax_line_kernel<P, T, false, F>})
      SEM_CUDA(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)C::SMEM));
    return true;
  }();
  (void)done;
}

template <int P, class T>
static void launch_line_p(const sem_handle* h, const OpData<T>& op, const T* u, T* w, T h1, T h2,
                          const T* h1f, bool fuse, const CGState* st, cudaStream_t s) {
  using C = LineCfg<P, T>;
  constexpr bool F = sizeof(T) == 4;
  auto kern = h1f ? (fuse ? ax_line_kernel<P, T, true, F> : ax_line_kernel<P, T, false, F>)
                  : (fuse ? ax_line_kernel<P, T, true, false> : ax_line_kernel<P, T, false, false>);
  configure_line<P, T>();
  DMat<P, T> D;
  for (int a = 0; a < P * P; ++a) D.d[a] = (T)h->Dh[a];
  const int E = (int)h->E;
  const FuseBox fb{h->nelx, h->nely, h->nelz, h->faces};
  kern<<<(E + C::K - 1) / C::K, C::THREADS, C::SMEM, s>>>(u, w, op.G.ptr, op.B.ptr, h1f, h1, h2, D,
                                                          op.D.ptr + P * P, E, fb, st);
  SEM_CHECK_LAUNCH();
}

template <class T>
void launch_ax_line(const sem_handle* h, const OpData<T>& op, const T* u, T* w, T h1, T h2,
                    const T* h1f, bool fuse, const CGState* st, cudaStream_t s) {
  if constexpr (sizeof(T) == 8) {
    if (h->P == 8) return launch_line_p<8, T>(h, op, u, w, h1, h2, h1f, fuse, st, s);
    if (h->P == 10) return launch_line_p<10, T>(h, op, u, w, h1, h2, h1f, fuse, st, s);
  } else {
    switch (h->P) {
      case 2: return launch_line_p<2, T>(h, op, u, w, h1, h2, h1f, fuse, st, s);
      case 3: return launch_line_p<3, T>(h, op, u, w, h1, h2, h1f, fuse, st, s);
      case 4: return launch_line_p<4, T>(h, op, u, w, h1, h2, h1f, fuse, st, s);
      case 5: return launch_line_p<5, T>(h, op, u, w, h1, h2, h1f, fuse, st, s);
      case 6: return launch_line_p<6, T>(h, op, u, w, h1, h2, h1f, fuse, st, s);
      case 7: return launch_line_p<7, T>(h, op, u, w, h1, h2, h1f, fuse, st, s);
      case 8: return launch_line_p<8, T>(h, op, u, w, h1, h2, h1f, fuse, st, s);
      case 9: return launch_line_p<9, T>(h, op, u, w, h1, h2, h1f, fuse, st, s);
      case 10: return launch_line_p<10, T>(h, op, u, w, h1, h2, h1f, fuse, st, s);
      case 11: return launch_line_p<11, T>(h, op, u, w, h1, h2, h1f, fuse, st, s);
    }
  }
  throw Error(SEM_ERR_ARG, "launch_ax_line: unsupported order");
}

void line_prepare(const sem_handle* h) {
  if (h->P == 8) configure_line<8, double>();
  if (h->P == 10) configure_line<10, double>();
  if (!h->f32.G.ptr) return;
  switch (h->P) {
    case 2: return configure_line<2, float>();
    case 3: return configure_line<3, float>();
    case 4: return configure_line<4, float>();
    case 5: return configure_line<5, float>();
    case 6: return configure_line<6, float>();
    case 7: return configure_line<7, float>();
    case 8: return configure_line<8, float>();
    case 9: return configure_line<9, float>();
    case 10: return configure_line<10, float>();
    case 11: return configure_line<11, float>();
  }
}

template void launch_ax_line<float>(const sem_handle*, const OpData<float>&, const float*, float*,
                                    float, float, const float*, bool, const CGState*,
                                    cudaStream_t);
template void launch_ax_line<double>(const sem_handle*, const OpData<double>&, const double*,
                                     double*, double, double, const double*, bool, const CGState*,
                                     cudaStream_t);

}  // namespace sem
