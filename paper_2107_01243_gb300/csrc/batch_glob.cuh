// The batched solver's FP32 inner PCG on global (unique-dof) vectors (the
// single-problem form is global.cu and cg.cu): per order class, one element
// launch over the elements of all problems of the class (the line kernel on
// global vectors; it also forms <p, H p> from the local products, p being
// continuous and zero on Dirichlet points), then per-problem-chunk vector
// kernels with plain dots that also clear w for the next operator.  Finished
// problems are stepped over.  Included by batch.cu (it needs BProb, item_sum,
// KahanF).
#pragma once

namespace sem {

// Element launch of one order class: CTA g takes the K consecutive elements
// groups[g] = (problem, first element) of one problem (ax_line.cuh), gathers
// and scatters as ax_glob_kernel (global.cu) and its warps add their
// shares of <p, H p> to the problem's accumulators.
template <int P>
__global__ void __launch_bounds__(LineCfg<P, float, kGlobThreads>::THREADS,
                                  LineCfg<P, float, kGlobThreads>::MINB)
bglob_kernel(const BProb* __restrict__ probs, const int2* __restrict__ groups,
             const __grid_constant__ DMat<P, float> D) {
  using C = LineCfg<P, float, kGlobThreads>;
  constexpr int P3 = C::P3, N = P - 1, NW = C::THREADS / 32;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  const int2 grp = __ldg(groups + blockIdx.x);
  const BProb& b = probs[grp.x];
  if (const int done = b.st->done) {       // finished (a pending x has been advanced)
    if (done == kXPending && grp.y == 0 && threadIdx.x == 0) b.st->done = 1;
    return;
  }
  LineThread<P, float, kGlobThreads> t;
  t.init(smem_raw);
  const int e = grp.y + t.el;
  const bool act = t.el < C::K && e < b.E;
  const int ee = act ? e : 0, sk = b.gx * b.gy;            // n_G < 2^31
  const uint32_t r1 = b.dnx.div((uint32_t)ee), ezu = b.dny.div(r1);
  const int ex = ee - (int)r1 * b.nelx, ey = (int)(r1 - ezu * (uint32_t)b.nely), ez = (int)ezu;
  const int org = ex * N + t.i + b.gx * (ey * N + t.j) + sk * (ez * N);
  const float* u = b.pg;
  float uc[P], out[P];
  if (act) {
#pragma unroll
    for (int k = 0; k < P; ++k) uc[k] = u[org + sk * k];
  }
  const size_t base = (size_t)ee * P3 + t.lam;
  line_element(t, act, D, uc, b.G + (size_t)ee * 6 * P3 + t.lam, b.B + base, (const float*)nullptr,
               b.h1, b.h2, out);
  float pw = 0.0f, pw_c = 0.0f;            // Kahan-compensated <p, H p>
  if (act) {
    int dst0 = org;                        // the column's addresses are made anew:
    asm volatile("" : "+r"(dst0));         // kept since the gather they would spill
    const int f = b.faces;
    const unsigned fl = ((f & SEM_FACE_XMIN) && ex == 0 ? 4u : 0u) |
                        ((f & SEM_FACE_XMAX) && ex == b.nelx - 1 ? 8u : 0u) |
                        ((f & SEM_FACE_YMIN) && ey == 0 ? 16u : 0u) |
                        ((f & SEM_FACE_YMAX) && ey == b.nely - 1 ? 32u : 0u) |
                        ((f & SEM_FACE_ZMIN) && ez == 0 ? 64u : 0u) |
                        ((f & SEM_FACE_ZMAX) && ez == b.nelz - 1 ? 128u : 0u);
    const bool fij = t.i == 0 || t.i == N || t.j == 0 || t.j == N;
    const unsigned pij = (t.i == 0 ? 4u : 0u) | (t.i == N ? 8u : 0u) | (t.j == 0 ? 16u : 0u) |
                         (t.j == N ? 32u : 0u);
    float* w = b.wg;
#pragma unroll
    for (int k = 0; k < P; ++k) {
      const float y = __fsub_rn(__fmul_rn(uc[k], out[k]), pw_c);
      const float tt = __fadd_rn(pw, y);
      pw_c = __fsub_rn(__fsub_rn(tt, pw), y);
      pw = tt;
      const unsigned pf = pij | (k == 0 ? 64u : 0u) | (k == N ? 128u : 0u);
      if (pf & fl) continue;               // Dirichlet point: stays zero
      float* dst = w + (dst0 + sk * k);
      if (fij || k == 0 || k == N)
        red_add(dst, out[k]);
      else
        *dst = out[k];
    }
  }
  const FxVal f = fx_warp_sum(pw, pw_c);
  if ((threadIdx.x & 31) == 0)
    atomicAdd(b.pwacc + (blockIdx.x * NW + (threadIdx.x >> 5)) % kBatchSlots,
              fx_round(f.m >> 32, (long long)(unsigned)f.m, f.e));
}

// ---- vector kernels on global vectors: items of kGChunk values of one
// problem (a quarter of the L-vector item: small problems still give every
// SM several blocks)

// Starts the inner solve of the problems owning global items [item0, item0 + count):
// one problem's few items leave most of the chip idle, so that the latency of an
// item's loads is the time (16-byte loads, four ahead: 18 us; 4-byte 45).
__global__ void __launch_bounds__(256)
bginit_kernel(const BProb* __restrict__ probs, const int* __restrict__ item_prob, int item0,
              int count, int nitems, double* partials, unsigned* tickets, double tol, int maxit) {
  for (int it = item0 + blockIdx.x; it < item0 + count; it += gridDim.x) {
    const int pi = item_prob[it];
    const BProb& b = probs[pi];
    const long long lo = (long long)(it - b.g_off) * kGChunk;
    const long long hi = min(lo + kGChunk, b.nGp);
    float4* p4 = reinterpret_cast<float4*>(b.pg + lo);
    float4* x4 = reinterpret_cast<float4*>(b.xg + lo);
    float4* w4 = reinterpret_cast<float4*>(b.wg + lo);
    const float4* r4 = reinterpret_cast<const float4*>(b.rg + lo);
    const float4* d4 = reinterpret_cast<const float4*>(b.dinvg + lo);
    const int n4 = (int)((hi - lo) >> 2);
    const float4 zero = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    KahanF rz, rr;
#pragma unroll 4
    for (int q = threadIdx.x; q < n4; q += blockDim.x) {
      const float4 r = r4[q], d = d4[q];
      const float4 z = make_float4(d.x * r.x, d.y * r.y, d.z * r.z, d.w * r.w);
      p4[q] = z;
      x4[q] = zero;
      w4[q] = zero;
      rz.add(__fmul_rn(r.x, z.x));
      rz.add(__fmul_rn(r.y, z.y));
      rz.add(__fmul_rn(r.z, z.z));
      rz.add(__fmul_rn(r.w, z.w));
      rr.add(__fmul_rn(r.x, r.x));
      rr.add(__fmul_rn(r.y, r.y));
      rr.add(__fmul_rn(r.z, r.z));
      rr.add(__fmul_rn(r.w, r.w));
    }
    double v[2] = {rz.value(), rr.value()}, tot[2];
    if (item_sum<2>(v, partials, it, b.g_off, b.g_cnt, &tickets[pi], tot, nitems) &&
        threadIdx.x == 0) {
      CGState* st = b.st;
      st->rz = tot[0];
      st->rr = tot[1];
      st->bb = tot[1];
      st->tol2 = tol * tol * tot[1];
      st->iter = 0;
      st->status = SEM_OK;
      st->maxit = maxit;
      st->alpha = st->beta = 0.0;
      st->done = (tot[1] <= st->tol2 || tot[1] == 0.0 || maxit <= 0) ? 1 : 0;
      for (int q = 0; q < kBatchSlots; ++q) b.pwacc[q] = 0.0;
    }
    __syncthreads();
  }
}

// the global items of a launch, finished problems stepped over
struct GItemWalk {
  int goff[kMaxBatch + 1];
  int done[kMaxBatch];
  // pending: a problem that finished in this iteration still counts as running
  __device__ __forceinline__ void load(const BProb* __restrict__ probs, int nprob, int nitems,
                                       bool pending) {
    for (int q = threadIdx.x; q < nprob; q += blockDim.x) {
      goff[q] = probs[q].g_off;
      const int dn = probs[q].st->done;
      done[q] = pending ? dn == 1 : dn != 0;
    }
    if (threadIdx.x == 0) goff[nprob] = nitems;
    __syncthreads();
  }
  __device__ __forceinline__ int next(const int* __restrict__ item_prob, int it, int stride,
                                      int nitems) const {
    while (it < nitems) {
      const int pi = item_prob[it];
      if (!done[pi]) break;
      it += (goff[pi + 1] - it + stride - 1) / stride * stride;
    }
    return it;
  }
};

__device__ __forceinline__ void gupd1(float& r, float w, float d, float alpha, KahanF& rz,
                                      KahanF& rr) {
  r -= alpha * w;
  const float z = d * r;
  rz.add(__fmul_rn(r, z));
  rr.add(__fmul_rn(r, r));
}

// alpha = <r, z> / the sum of pwacc (the element kernel accumulated <p, H p>); the
// problem's last item block checks it, records it and clears the accumulator
__global__ void __launch_bounds__(256)
bgupdate_kernel(const BProb* __restrict__ probs, const int* __restrict__ item_prob, int nprob,
                int nitems, double* partials, unsigned* tickets) {
  __shared__ GItemWalk wk;
  wk.load(probs, nprob, nitems, false);
  for (int it = wk.next(item_prob, blockIdx.x, gridDim.x, nitems); it < nitems;
       it = wk.next(item_prob, it + gridDim.x, gridDim.x, nitems)) {
    const int pi = item_prob[it];
    const BProb& b = probs[pi];
    __shared__ FxVal sw[8];
    const double pwv = fx_block_total<8>(__ldcg(b.pwacc + threadIdx.x), sw);
    const float alpha = (float)(b.st->rz / pwv);
    const long long lo = (long long)(it - b.g_off) * kGChunk;
    const long long hi = min(lo + kGChunk, b.nGp);
    float4* r4 = reinterpret_cast<float4*>(b.rg + lo);
    float4* w4 = reinterpret_cast<float4*>(b.wg + lo);
    const float4* d4 = reinterpret_cast<const float4*>(b.dinvg + lo);
    const int n4 = (int)((hi - lo) >> 2);
    const float4 zero = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    KahanF rz, rr;
#pragma unroll 2
    for (int q = threadIdx.x; q < n4; q += blockDim.x) {
      float4 r = r4[q];
      const float4 w = w4[q], d = d4[q];
      gupd1(r.x, w.x, d.x, alpha, rz, rr);
      gupd1(r.y, w.y, d.y, alpha, rz, rr);
      gupd1(r.z, w.z, d.z, alpha, rz, rr);
      gupd1(r.w, w.w, d.w, alpha, rz, rr);
      r4[q] = r;
      w4[q] = zero;
    }
    double v[2] = {rz.value(), rr.value()}, tot[2];
    if (item_sum<2>(v, partials, it, b.g_off, b.g_cnt, &tickets[pi], tot, nitems)) {
      b.pwacc[threadIdx.x] = 0.0;
      if (threadIdx.x == 0) {
        CGState* st = b.st;
        st_after_pw(st, pwv);                // breakdown when <p, H p> <= 0
        if (!st->done) st_after_update(st, tot, kXPending);
      }
    }
    __syncthreads();
  }
}

__global__ void __launch_bounds__(256)
bgpupd_kernel(const BProb* __restrict__ probs, const int* __restrict__ item_prob, int nprob,
              int nitems) {
  __shared__ GItemWalk wk;
  wk.load(probs, nprob, nitems, true);
  for (int it = wk.next(item_prob, blockIdx.x, gridDim.x, nitems); it < nitems;
       it = wk.next(item_prob, it + gridDim.x, gridDim.x, nitems)) {
    const int pi = item_prob[it];
    const BProb& b = probs[pi];
    const bool last = b.st->done != 0;       // x only: no further direction
    const float alpha = (float)b.st->alpha, beta = (float)b.st->beta;
    const long long lo = (long long)(it - b.g_off) * kGChunk;
    const long long hi = min(lo + kGChunk, b.nGp);
    float4* p4 = reinterpret_cast<float4*>(b.pg + lo);
    float4* x4 = reinterpret_cast<float4*>(b.xg + lo);
    const float4* r4 = reinterpret_cast<const float4*>(b.rg + lo);
    const float4* d4 = reinterpret_cast<const float4*>(b.dinvg + lo);
    const int n4 = (int)((hi - lo) >> 2);
#pragma unroll 4
    for (int q = threadIdx.x; q < n4; q += blockDim.x) {
      float4 p = p4[q], x = x4[q];
      x.x += alpha * p.x;
      x.y += alpha * p.y;
      x.z += alpha * p.z;
      x.w += alpha * p.w;
      x4[q] = x;
      if (last) continue;
      const float4 r = r4[q], d = d4[q];
      p.x = d.x * r.x + beta * p.x;
      p.y = d.y * r.y + beta * p.y;
      p.z = d.z * r.z + beta * p.z;
      p.w = d.w * r.w + beta * p.w;
      p4[q] = p;
    }
  }
}

}  // namespace sem
