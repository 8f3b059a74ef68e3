// The assembled operator w = mask o QQ^T (h1 A_L + h2 B_L) u (arXiv 2107.01243
// §2, Eq. 9-10) with the gather-scatter split by direction.  On the box,
// QQ^T is the product of three commuting pair sums, one per direction: the
// copies of a point on an x-interface are the i = N value of element e and
// the i = 0 value of element e + 1, and so on for y (e + nelx) and z
// (e + nelx nely).  Summing the x-pairs, then the y-pairs, then the z-pairs
// gives every copy the sum of all its copies (2, 4 or 8).
//
//   local   the element kernel sums the x-pairs inside a segment of consecutive
//           elements itself (streaming kernels: kFuseSeg elements a CTA walks, the
//           upper one reading back the copy the lower one stored just before; the
//           line kernel: the elements of a CTA, through shared memory); masked
//           points are written as zero
//   finish  small vectors: k_finish, all remaining pairs in one pass; else
//           k_sx_cut: x-pairs between segments;
//           k_sy, k_sz: the y- and z-pairs, each a coalesced sweep over the
//           j = N / k = N planes of the elements and their neighbours' j = 0 /
//           k = 0 planes
//
// IEEE FP64 but for large meshes at N = 7 and 9: the element kernel of sem_ax, then
// the gather-scatter of sem_dssum.
//
// The x-face copies are 8-byte values 64 bytes apart (P = 8), so a separate
// gather-scatter spends a 32-byte sector on each; here they never leave the
// element kernel.  Summation order: ((x-pairs) + (x-pairs)) + ..., i.e. the
// copies of an edge point are added as (w0 + w1) + (w2 + w3); sem_dssum keeps
// the increasing-index order instead.
#include "sem_internal.cuh"
#include <type_traits>

#include "ax_line.cuh"
#include "ax_tile.cuh"

namespace sem {

bool launch_ax_tma_fused(const sem_handle* h, const float* u, float* w, float h1, float h2,
                         const float* h1f, const CGState* st, CGState* pwst, cudaStream_t s);
bool launch_ax_df_fused(const sem_handle* h, const double* u, double* w, double h1, double h2,
                        const CGState* st, CGState* pwst, cudaStream_t s);
void launch_ax_df_fused_slab(const sem_handle* h, const double* u, double* w, double h1,
                             double h2, int z0, int z1, cudaStream_t s);
bool df_ax_supported(const sem_handle* h, const void* u, const void* w, const void* h1f);

namespace {

// x-pairs at the segment starts of the element kernel: the first element
// e_b = g SEG of segment g >= 1 pairs its i = 0 face with the i = N face
// of the element before it, unless it starts an x-row.  Threads run over
// (j, k, segment start).
template <int P, int SEG, class T>
__global__ void __launch_bounds__(256)
k_sx_cut(T* __restrict__ w, uint32_t total, FastDiv dnx, const CGState* __restrict__ st) {
  if (st && st->done) return;
  constexpr uint32_t P2 = P * P;
  constexpr long long P3 = (long long)P2 * P;
  for (uint32_t t = blockIdx.x * blockDim.x + threadIdx.x; t < total;
       t += gridDim.x * blockDim.x) {
    const uint32_t c = t / P2, jk = t - c * P2, eb = (c + 1) * SEG;
    if (eb == dnx.div(eb) * dnx.d) continue;
    const long long hi = (long long)eb * P3 + (long long)jk * P;   // (eb, 0, j, k)
    const long long lo = hi - P3 + (P - 1);                         // (eb - 1, N, j, k)
    const T sum = w[lo] + w[hi];
    w[lo] = sum;
    w[hi] = sum;
  }
}

// VW values of T moved together
template <class T, int VW>
struct alignas(VW * sizeof(T)) Pack {
  T v[VW];
};

// y-pairs: (e, i, N, k) + (e + nelx, i, 0, k) for every element with
// ey < nely - 1; a thread takes VW neighbouring i (VW divides P, w aligned to
// VW values), threads run over (i, k, element) with i fastest
template <int P, int VW, class T>
__global__ void __launch_bounds__(256)
k_sy(T* __restrict__ w, int nelx, int nely, uint32_t total, FastDiv dnx, FastDiv dny1,
     const CGState* __restrict__ st) {
  if (st && st->done) return;
  constexpr int H = P / VW, P2 = P * P, P3 = P2 * P;
  using V = Pack<T, VW>;
  V* wv = reinterpret_cast<V*>(w);
  for (uint32_t t = blockIdx.x * blockDim.x + threadIdx.x; t < total;
       t += gridDim.x * blockDim.x) {
    const uint32_t ip = t % H, r = t / H;
    const uint32_t k = r % P, m = r / P;            // element among those with ey < nely - 1
    const uint32_t r2 = dnx.div(m);
    const uint32_t ex = m - r2 * (uint32_t)nelx;
    const uint32_t ez = dny1.div(r2);
    const uint32_t ey = r2 - ez * (uint32_t)(nely - 1);
    const uint32_t e = ex + (uint32_t)nelx * (ey + (uint32_t)nely * ez);
    const uint32_t lo = (e * P3 + k * P2 + (P - 1) * P) / VW + ip;
    const uint32_t hi = ((e + nelx) * P3 + k * P2) / VW + ip;
    V a = wv[lo];
    const V b = wv[hi];
#pragma unroll
    for (int c = 0; c < VW; ++c) a.v[c] = a.v[c] + b.v[c];
    wv[lo] = a;
    wv[hi] = a;
  }
}

// z-pairs: (e, i, j, N) + (e + nelx nely, i, j, 0) for every element with
// ez < nelz - 1 (the first nelx nely (nelz - 1) elements), VW values a thread
// (VW divides P^2, w aligned to VW values)
template <int P, int VW, class T>
__global__ void __launch_bounds__(256)
k_sz(T* __restrict__ w, uint32_t layer, uint32_t total, const CGState* __restrict__ st) {
  if (st && st->done) return;
  constexpr int P2 = P * P, P3 = P2 * P, Q = P2 / VW;
  using V = Pack<T, VW>;
  V* wv = reinterpret_cast<V*>(w);
  for (uint32_t t = blockIdx.x * blockDim.x + threadIdx.x; t < total;
       t += gridDim.x * blockDim.x) {
    const uint32_t q = t % Q, e = t / Q;
    const uint32_t lo = (e * P3 + (P - 1) * P2) / VW + q;
    const uint32_t hi = ((e + layer) * P3) / VW + q;
    V a = wv[lo];
    const V b = wv[hi];
#pragma unroll
    for (int c = 0; c < VW; ++c) a.v[c] = a.v[c] + b.v[c];
    wv[lo] = a;
    wv[hi] = a;
  }
}

int sweep_blocks(long long total) {
  return (int)std::max<long long>(1, std::min<long long>((total + 255) / 256, 16LL * sem_num_sms()));
}

// whether w starts on a multiple of VW values (element bases are then too: VW
// divides P^2)
template <int VW, class T>
bool aligned_to(const T* w) {
  return reinterpret_cast<uintptr_t>(w) % (VW * sizeof(T)) == 0;
}

template <int P, class T>
void launch_sy(T* w, int nelx, int nely, int nelz, const CGState* st, cudaStream_t s) {
  auto go = [&](auto vw) {
    constexpr int VW = decltype(vw)::value;
    const long long total = (long long)nelx * (nely - 1) * nelz * P * (P / VW);
    k_sy<P, VW, T><<<sweep_blocks(total), 256, 0, s>>>(w, nelx, nely, (uint32_t)total,
                                                       FastDiv((uint32_t)nelx),
                                                       FastDiv((uint32_t)(nely - 1)), st);
    SEM_CHECK_LAUNCH();
  };
  if constexpr (P % 2 == 0)
    if (aligned_to<2>(w)) return go(std::integral_constant<int, 2>());
  go(std::integral_constant<int, 1>());
}

// the z-pairs of nz element layers and the ones above them
template <int P, class T>
void launch_sz(T* w, long long layer, int nz, const CGState* st, cudaStream_t s) {
  auto go = [&](auto vw) {
    constexpr int VW = decltype(vw)::value;
    const long long total = layer * nz * P * P / VW;
    k_sz<P, VW, T><<<sweep_blocks(total), 256, 0, s>>>(w, (uint32_t)layer, (uint32_t)total, st);
    SEM_CHECK_LAUNCH();
  };
  constexpr int W = 16 / (int)sizeof(T);
  if constexpr (P * P % W == 0)
    if (aligned_to<W>(w)) return go(std::integral_constant<int, W>());
  go(std::integral_constant<int, 1>());
}

// All the pairs the element kernel left, in one pass: every point on a z-face
// between elements (Z), on a y-face but no such z-face (Y), on an x-face between
// segments but neither (X).  A thread owns all the copies of its
// point (the lowest copy's place tells it) and sums them pair by pair along x,
// y, z; the x-pairs inside a segment already agree, so one of the two is read
// and both are written.  Threads run over (i, j) or
// (i, k) of an element, i fastest.
template <int P, int SEG, class T>
__global__ void __launch_bounds__(256)
k_finish(T* __restrict__ w, int nelx, int nely, int nelz, uint32_t nZ, uint32_t nY, uint32_t nX,
         FastDiv dnx, FastDiv dny, FastDiv dny1, const CGState* __restrict__ st) {
  if (st && st->done) return;
  constexpr int N = P - 1, P2 = P * P, P3 = P2 * P;
  const uint32_t total = nZ + nY + nX;
  for (uint32_t t = blockIdx.x * blockDim.x + threadIdx.x; t < total;
       t += gridDim.x * blockDim.x) {
    uint32_t e;
    int i, j, k, ex, ey, ez;
    if (t < nZ) {
      e = t / P2;
      const int q = (int)(t - e * P2);
      i = q % P;
      j = q / P;
      k = N;
      const uint32_t r = dnx.div(e);
      ex = (int)(e - r * (uint32_t)nelx);
      ez = (int)dny.div(r);
      ey = (int)r - ez * nely;
      if (j == 0 && ey > 0) continue;                       // its row j = N below owns it
    } else if (t < nZ + nY) {
      const uint32_t m = (t - nZ) / P2;                     // elements with ey < nely - 1
      const int q = (int)((t - nZ) - m * P2);
      i = q % P;
      j = N;
      k = q / P;
      const uint32_t r = dnx.div(m);
      ex = (int)(m - r * (uint32_t)nelx);
      ez = (int)dny1.div(r);
      ey = (int)r - ez * (nely - 1);
      e = (uint32_t)(ex + nelx * (ey + nely * ez));
      if ((k == 0 && ez > 0) || (k == N && ez < nelz - 1)) continue;   // on a z-face
    } else {
      const uint32_t c = (t - nZ - nY) / P2;
      const int q = (int)((t - nZ - nY) - c * P2);
      e = (c + 1) * SEG - 1;                                // last of its segment
      i = N;
      j = q % P;
      k = q / P;
      const uint32_t r = dnx.div(e);
      ex = (int)(e - r * (uint32_t)nelx);
      ez = (int)dny.div(r);
      ey = (int)r - ez * nely;
      if (ex == nelx - 1 || (j == 0 && ey > 0) || (j == N && ey < nely - 1) ||
          (k == 0 && ez > 0) || (k == N && ez < nelz - 1))
        continue;
    }
    if (i == 0 && ex > 0) continue;                         // e - 1's column i = N owns it
    const bool fx = i == N && ex < nelx - 1, fy = j == N && ey < nely - 1,
               fz = k == N && ez < nelz - 1;
    const int ox = P3 - N, oy = nelx * P3 - N * P, oz = nelx * nely * P3 - N * P2;
    T* const b = w + ((size_t)e * P3 + (k * P + j) * P + i);
    // FP64: adds that no lane of the warp needs are skipped (a warp's FP64 add
    // takes 64 cycles of a scheduler, predicated or not)
    bool anyy = fy, anyz = fz;
    if constexpr (sizeof(T) == 8) {
      const unsigned am = __activemask();
      anyy = __any_sync(am, fy);
      anyz = __any_sync(am, fz);
    }
    // the (y, z) copies; at a segment end the x-partner's value is still apart
    T c[4], x[4];
    bool cut[4];
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      const bool in = (!(m & 1) || fy) && (!(m & 2) || fz);
      const int o = ((m & 1) ? oy : 0) + ((m & 2) ? oz : 0);
      const uint32_t em = e + ((m & 1) ? (uint32_t)nelx : 0u) + ((m & 2) ? (uint32_t)(nelx * nely) : 0u);
      cut[m] = in && fx && (em + 1) % SEG == 0;
      c[m] = in ? b[o] : T(0);
      x[m] = cut[m] ? b[o + ox] : T(0);
    }
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      bool any = cut[m];
      if constexpr (sizeof(T) == 8) any = __any_sync(__activemask(), cut[m]);
      if (any) c[m] += x[m];               // x = 0 where there is no cut
    }
    T s = c[0];
    if (anyy) s += c[1];                   // 0 where there is no copy
    if (anyz) {
      T s2 = c[2];
      if (anyy) s2 += c[3];
      s += s2;
    }
#pragma unroll
    for (int m = 0; m < 4; ++m)
      if ((!(m & 1) || fy) && (!(m & 2) || fz)) {
        const int o = ((m & 1) ? oy : 0) + ((m & 2) ? oz : 0);
        b[o] = s;
        if (fx) b[o + ox] = s;
      }
  }
}

// Up to this many bytes of w one pass over the shared points takes the place of
// the three: it saves two launches, but its copies across an x-face are
// scattered writes that cost more than the launches once w no longer sits in
// the caches.  FP32 (finish alone, us, one pass / three): N = 7, 0.9 M points 11 / 14,
// 4.1 M 11 / 15, 16.8 M 30 / 24.  FP64, whose pass also pays for the adds on the FP64
// pipe (sem_apply): N = 7, 7.1 MB 31.4 / 32.0, 11.2 MB 44.3 / 43.3, 16.8 MB
// 61.8 / 59.1; N = 5, 4.7 MB 26.5 / 27.1, 7.1 MB 37.0 / 36.7, 13.8 MB 62.1 / 59.0.
template <class T>
constexpr long long kOnePassBytes = sizeof(T) == 8 ? 7 << 20 : 1 << 24;

// the finishing passes on a box of nelx x nely x nelz elements starting at w,
// after an element kernel with segments of SEG elements
template <int P, int SEG, class T>
void finish_box(T* w, int nelx, int nely, int nelz, const CGState* st, cudaStream_t s) {
  const long long layer = (long long)nelx * nely, E = layer * nelz, P2 = P * P;
  const long long nX = nelx > 1 ? ((E + SEG - 1) / SEG - 1) * P2 : 0;
  if (E * P2 * P * (long long)sizeof(T) <= kOnePassBytes<T>) {
    const long long nZ = layer * (nelz - 1) * P2, nY = (long long)nelx * (nely - 1) * nelz * P2;
    if (nZ + nY + nX == 0) return;
    const int blocks = (int)std::min<long long>((nZ + nY + nX + 255) / 256, 64LL * sem_num_sms());
    k_finish<P, SEG, T><<<blocks, 256, 0, s>>>(
        w, nelx, nely, nelz, (uint32_t)nZ, (uint32_t)nY, (uint32_t)nX, FastDiv((uint32_t)nelx),
        FastDiv((uint32_t)nely), FastDiv((uint32_t)std::max(1, nely - 1)), st);
    SEM_CHECK_LAUNCH();
    return;
  }
  if (nX > 0) {
    k_sx_cut<P, SEG, T><<<sweep_blocks(nX), 256, 0, s>>>(w, (uint32_t)nX, FastDiv((uint32_t)nelx),
                                                         st);
    SEM_CHECK_LAUNCH();
  }
  if (nely > 1) launch_sy<P, T>(w, nelx, nely, nelz, st, s);
  if (nelz > 1) launch_sz<P, T>(w, layer, nelz - 1, st, s);
}

// z-pairs between element planes z - 1 and z of the box (one plane of pairs)
template <int P, class T>
void zpairs_between(const sem_handle* h, T* w, int z, cudaStream_t s) {
  constexpr long long P3 = (long long)P * P * P;
  const long long layer = (long long)h->nelx * h->nely;
  launch_sz<P, T>(w + (z - 1) * layer * P3, layer, 1, nullptr, s);
}

// the finishing passes of the slab of element planes [z0, z1), then (z0 > 0)
// the z-pairs between it and the slab below
template <int P>
void finish_slab(const sem_handle* h, double* w, int z0, int z1, cudaStream_t s) {
  constexpr long long P3 = (long long)P * P * P;
  finish_box<P, kFuseSeg, double>(w + (long long)z0 * h->nelx * h->nely * P3, h->nelx, h->nely, z1 - z0,
                        nullptr, s);
  if (z0 > 0) zpairs_between<P, double>(h, w, z0, s);
}

// line: the element kernel was the line kernel (its own segment length)
template <int P, class T>
void finish_p(const sem_handle* h, T* w, bool line, const CGState* st, cudaStream_t s) {
  if constexpr (sizeof(T) == 4 || eo_split(P, true))
    if (line)
      return finish_box<P, line_elems(P, sizeof(T) == 8), T>(w, h->nelx, h->nely, h->nelz, st, s);
  if constexpr (P % 2 == 0) finish_box<P, kFuseSeg, T>(w, h->nelx, h->nely, h->nelz, st, s);
}

template <class T>
void finish(const sem_handle* h, T* w, bool line, const CGState* st, cudaStream_t s) {
  switch (h->P) {
    case 2: finish_p<2, T>(h, w, line, st, s); break;
    case 3: finish_p<3, T>(h, w, line, st, s); break;
    case 4: finish_p<4, T>(h, w, line, st, s); break;
    case 5: finish_p<5, T>(h, w, line, st, s); break;
    case 6: finish_p<6, T>(h, w, line, st, s); break;
    case 7: finish_p<7, T>(h, w, line, st, s); break;
    case 8: finish_p<8, T>(h, w, line, st, s); break;
    case 9: finish_p<9, T>(h, w, line, st, s); break;
    case 10: finish_p<10, T>(h, w, line, st, s); break;
    case 11: finish_p<11, T>(h, w, line, st, s); break;
    default: throw Error(SEM_ERR_ARG, "apply: unsupported order");
  }
}

}  // namespace

template <>
bool apply_fused_supported<float>(const sem_handle* h, const void* u, const void* w,
                                  const void* h1f) {
  return h->f32.G.ptr && tma_ax_supported<float>(h, u, w, h1f) && h->nL < (1LL << 31);
}

template <>
bool apply_fused_supported<double>(const sem_handle* h, const void* u, const void* w,
                                   const void* h1f) {
  return h->f64_kernel != SEM_F64_KERNEL_NATIVE && df_ax_supported(h, u, w, h1f) &&
         h->nL < (1LL << 31);
}

template <class T>
bool launch_apply(sem_handle* h, const OpData<T>& op, const T* u, T* w, T h1, T h2, const T* h1f,
                  const CGState* st, int phase, cudaStream_t s, CGState* pwst) {
  // the streaming kernels (double-float; FP32 bulk copies where they are tuned,
  // or asked for <p, H p>), else the line kernel, else element kernel and
  // gather-scatter (the FP64 orders and errors of launch_ax)
  bool stream = apply_fused_supported<T>(h, u, w, h1f);
  if (sizeof(T) == 4) stream = stream && (!h->tune.ax32_ldg || (pwst && h->P == 8));
  if (!stream) {
    const bool line = line_ax_supported<T>(h) && h->nL < (1LL << 31);
    if (phase & SEM_APPLY_LOCAL) {
      if (line) launch_ax_line<T>(h, op, u, w, h1, h2, h1f, true, st, s);
      else launch_ax<T>(h, op, u, w, h1, h2, h1f, st, s);
    }
    if (phase & SEM_APPLY_FINISH) {
      if (line) finish<T>(h, w, true, st, s);
      else launch_dssum<T>(h, w, true, st, s);
    }
    return false;
  }
  bool pw = false;
  if (phase & SEM_APPLY_LOCAL) {
    if constexpr (std::is_same<T, float>::value)
      pw = launch_ax_tma_fused(h, u, w, h1, h2, h1f, st, pwst, s);
    else
      pw = launch_ax_df_fused(h, u, w, h1, h2, st, pwst, s);
  }
  if (phase & SEM_APPLY_FINISH) finish<T>(h, w, false, st, s);
  return pw;
}

// Streams and events of the pipelined host-buffer operator, kept per handle.
struct HostPipe {
  static constexpr int kSlabs = 8;
  cudaStream_t in = nullptr, comp = nullptr, out = nullptr;
  cudaEvent_t start = nullptr, arrived[kSlabs] = {}, final_[kSlabs] = {};
  HostPipe() {
    SEM_CUDA(cudaStreamCreateWithFlags(&in, cudaStreamNonBlocking));
    SEM_CUDA(cudaStreamCreateWithFlags(&comp, cudaStreamNonBlocking));
    SEM_CUDA(cudaStreamCreateWithFlags(&out, cudaStreamNonBlocking));
    SEM_CUDA(cudaEventCreateWithFlags(&start, cudaEventDisableTiming));
    for (int q = 0; q < kSlabs; ++q) {
      SEM_CUDA(cudaEventCreateWithFlags(&arrived[q], cudaEventDisableTiming));
      SEM_CUDA(cudaEventCreateWithFlags(&final_[q], cudaEventDisableTiming));
    }
  }
  ~HostPipe() {
    for (int q = 0; q < kSlabs; ++q) {
      if (arrived[q]) cudaEventDestroy(arrived[q]);
      if (final_[q]) cudaEventDestroy(final_[q]);
    }
    if (start) cudaEventDestroy(start);
    for (cudaStream_t t : {in, comp, out})
      if (t) cudaStreamDestroy(t);
  }
};

bool host_pipeline_supported(const sem_handle* h, const void* din, const void* dout) {
  return h->nelz >= 2 && apply_fused_supported<double>(h, din, dout, nullptr);
}

// w_host = mask o QQ^T A_L u_host (FP64) with the copies overlapped with the
// work: the box is cut into slabs of element planes; slab q is copied in on
// one stream, its element kernel and finishing passes (and the z-pairs with
// slab q - 1) run on a second, and the planes those passes made final are
// copied out on a third while later slabs are still arriving or being
// computed.  Every pair sum is the one the unsplit operator forms, so the
// result is the same.
void apply_host_pipelined(sem_handle* h, const double* u_host, double* w_host, double* din,
                          double* dout, cudaStream_t user) {
  if (!h->host_pipe) h->host_pipe = std::make_shared<HostPipe>();
  HostPipe& hp = *h->host_pipe;
  const int S = std::min(HostPipe::kSlabs, h->nelz);
  const long long P3 = h->P3, layer = (long long)h->nelx * h->nely;
  std::vector<int> z(S + 1);
  for (int q = 0; q <= S; ++q) z[q] = (int)((long long)q * h->nelz / S);
  SEM_CUDA(cudaEventRecord(hp.start, user));
  SEM_CUDA(cudaStreamWaitEvent(hp.in, hp.start, 0));
  SEM_CUDA(cudaStreamWaitEvent(hp.comp, hp.start, 0));
  SEM_CUDA(cudaStreamWaitEvent(hp.out, hp.start, 0));
  for (int q = 0; q < S; ++q) {
    const long long o = z[q] * layer * P3, n = (long long)(z[q + 1] - z[q]) * layer * P3;
    SEM_CUDA(cudaMemcpyAsync(din + o, u_host + o, n * sizeof(double), cudaMemcpyHostToDevice,
                             hp.in));
    SEM_CUDA(cudaEventRecord(hp.arrived[q], hp.in));
  }
  for (int q = 0; q < S; ++q) {
    SEM_CUDA(cudaStreamWaitEvent(hp.comp, hp.arrived[q], 0));
    launch_ax_df_fused_slab(h, din, dout, 1.0, 0.0, z[q], z[q + 1], hp.comp);
    switch (h->P) {
      case 6: finish_slab<6>(h, dout, z[q], z[q + 1], hp.comp); break;
      case 8: finish_slab<8>(h, dout, z[q], z[q + 1], hp.comp); break;
      case 10: finish_slab<10>(h, dout, z[q], z[q + 1], hp.comp); break;
      default: throw Error(SEM_ERR_ARG, "apply_host_pipelined: unsupported order");
    }
    SEM_CUDA(cudaEventRecord(hp.final_[q], hp.comp));
  }
  // after slab q's passes the planes from the last plane of slab q - 1 up to
  // (not including) slab q's last plane are final; the last slab's last
  // plane too
  for (int q = 0; q < S; ++q) {
    const long long p0 = q == 0 ? z[0] : z[q] - 1, p1 = q == S - 1 ? z[S] : z[q + 1] - 1;
    if (p1 <= p0) continue;
    const long long o = p0 * layer * P3, n = (p1 - p0) * layer * P3;
    SEM_CUDA(cudaStreamWaitEvent(hp.out, hp.final_[q], 0));
    SEM_CUDA(cudaMemcpyAsync(w_host + o, dout + o, n * sizeof(double), cudaMemcpyDeviceToHost,
                             hp.out));
  }
  SEM_CUDA(cudaStreamSynchronize(hp.out));
  SEM_CUDA(cudaStreamSynchronize(hp.comp));
}

template bool launch_apply<float>(sem_handle*, const OpData<float>&, const float*, float*, float,
                                  float, const float*, const CGState*, int, cudaStream_t,
                                  CGState*);
template bool launch_apply<double>(sem_handle*, const OpData<double>&, const double*, double*,
                                   double, double, const double*, const CGState*, int,
                                   cudaStream_t, CGState*);

}  // namespace sem

using namespace sem;

extern "C" sem_status sem_apply(sem_handle* h, const void* u_L, void* w_L, double h1, double h2,
                                const void* h1_field, int dtype, int phase, void* stream) {
  return guarded("sem_apply", [&] {
    SEM_REQUIRE(h && u_L && w_L, "sem_apply: null argument");
    SEM_REQUIRE(phase == SEM_APPLY_FULL || phase == SEM_APPLY_LOCAL || phase == SEM_APPLY_FINISH,
                "sem_apply: phase must be SEM_APPLY_FULL, _LOCAL or _FINISH");
    SEM_REQUIRE(u_L != w_L, "sem_apply: u and w must not alias");
    cudaStream_t s = (cudaStream_t)stream;
    if (dtype == SEM_F64) {
      SEM_REQUIRE(h->f64.G.ptr, "sem_apply: handle has no FP64 geometry");
      launch_apply<double>(h, h->f64, (const double*)u_L, (double*)w_L, h1, h2,
                           (const double*)h1_field, nullptr, phase, s);
    } else if (dtype == SEM_F32) {
      SEM_REQUIRE(h->f32.G.ptr, "sem_apply: handle has no FP32 geometry");
      launch_apply<float>(h, h->f32, (const float*)u_L, (float*)w_L, (float)h1, (float)h2,
                          (const float*)h1_field, nullptr, phase, s);
    } else {
      throw Error(SEM_ERR_ARG, "sem_apply: dtype must be SEM_F64 or SEM_F32");
    }
  });
}
