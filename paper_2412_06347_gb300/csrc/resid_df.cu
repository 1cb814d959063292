// Residual update of the defect correction, r <- r - s D e per RHS: D applied in
// double-float arithmetic (df.cuh) to the exact FP32 values of e, on the FP64
// links and clover split once into FP32 (hi, lo) words.
//
// What bounds it: FP32 issue and instruction fetch.  D is about 1130
// double-float operations of 11 to 15 FP32 instructions per site; unrolled over
// the eight hops that is some 14 K instructions of straight-line code, which ran
// at 28 % of the issue rate with 12 warps per SM (42.6 ms at 64x32^3, 16 RHS).
// Here the two half-spinor components of a hop, which meet the same link, are
// the lanes of packed FP32 pairs, so one instruction does both, and the hops are
// a rolled loop (together 25.0 ms) whose spin structure is data: with e_0 = -1 and e_k = -i sigma_k,
//     h = u - s tau . i^im . swap(l),  lower += s sigma . i^im . swap(g)
// over the pair of spins, im = 1 for mu = 1, 3, swap for mu = 1, 2, tau = (1, 1),
// (1, 1), (1, -1), (1, -1) and sigma = tau but for sigma_0 = -tau_0.  The factors
// -1/2 and the time-boundary sign are exact and ride on the final sum and on h.
#include "internal.h"
#include "stencil.cuh"

namespace mglma {
namespace {

// packed FP32 pairs; the double-float operations on them are df.cuh's
__device__ __forceinline__ float2 pmul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 pdup(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 pswap(float2 a, bool s) { return s ? make_float2(a.y, a.x) : a; }
__device__ __forceinline__ float2 pneg(float2 a) { return make_float2(-a.x, -a.y); }

struct CD2 {
  DF2 re, im;
};

}  // namespace

__global__ void __launch_bounds__(128, 3) resid_df_kernel(const float4* __restrict__ e, double2* __restrict__ r,
                                                          const float4* __restrict__ U, const float4* __restrict__ C,
                                                          LatIdx q, float bc, int nrhs, const double* __restrict__ scale) {
  const int64_t V = q.V;
  // RHS fastest: the CTAs that share a block of sites are resident together
  const int64_t site = (int64_t)(blockIdx.x / nrhs) * blockDim.x + threadIdx.x;
  const int rhs = (int)(blockIdx.x % nrhs);
  if (site >= V) return;
  int x[4];
  site_coords(q, site, x);
  const float4* er = e + (size_t)rhs * 6 * V;
  const DF2 zero;
  CD2 up[3], lw[3];  // sums of the hops over spins (0, 1) and (2, 3), per colour
#pragma unroll
  for (int c = 0; c < 3; ++c) up[c] = lw[c] = CD2{zero, zero};
#pragma unroll 1
  for (int h = 0; h < 8; ++h) {
    const int mu = h >> 1;
    const bool fwd = !(h & 1);
    const int xm = mu == 0 ? x[0] : mu == 1 ? x[1] : mu == 2 ? x[2] : x[3];
    const int L = q.L[mu];
    const int64_t S = q.S[mu];
    const bool wrap = fwd ? xm == L - 1 : xm == 0;
    const int64_t n = site + (fwd ? (wrap ? -(int64_t)(L - 1) * S : S) : (wrap ? (int64_t)(L - 1) * S : -S));
    const float s = fwd ? -1.f : 1.f;  // (1 + s gamma_mu)
    const bool im = mu & 1, sw = mu == 1 || mu == 2;
    const float2 tau = make_float2(1.f, mu >= 2 ? -1.f : 1.f);
    const float bs = mu == 0 && wrap ? bc : 1.f;
    // projection: exact sums of two FP32 values
    CD2 hp[3];
    {
      float4 p[6];
#pragma unroll
      for (int j = 0; j < 6; ++j) p[j] = __ldg(er + (size_t)j * V + n);
      auto comp = [&](int k) { return k & 1 ? make_float2(p[k / 2].z, p[k / 2].w) : make_float2(p[k / 2].x, p[k / 2].y); };
      const float2 f = pmul(pdup(-s), tau);
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const float2 u0 = comp(c), u1 = comp(3 + c), l0 = comp(6 + c), l1 = comp(9 + c);
        const float2 lr = pswap(make_float2(l0.x, l1.x), sw), li = pswap(make_float2(l0.y, l1.y), sw);
        const float2 tr = im ? make_float2(-li.x, -li.y) : lr, ti = im ? lr : li;
        hp[c].re = dfl::two_sum(pmul(pdup(bs), make_float2(u0.x, u1.x)), pmul(pmul(pdup(bs), f), tr));
        hp[c].im = dfl::two_sum(pmul(pdup(bs), make_float2(u0.y, u1.y)), pmul(pmul(pdup(bs), f), ti));
      }
    }
    const float4* ul = U + (size_t)mu * 9 * V + (fwd ? site : n);
    const float sg = fwd ? 1.f : -1.f;  // U^dag: rows and columns exchanged, conjugated
    const int ra = fwd ? 3 : 1, rb = fwd ? 1 : 3;
    float2 sl = pmul(pdup(s), tau);
    if (mu == 0) sl = pmul(pdup(-1.f), sl);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      CD2 g{zero, zero};
#pragma unroll
      for (int b = 0; b < 3; ++b) {
        const float4 w = __ldg(ul + (size_t)(a * ra + b * rb) * V);  // re.hi, re.lo, im.hi, im.lo
        const float2 rh = pdup(w.x), rl = pdup(w.y), ih = pdup(sg * w.z), il = pdup(sg * w.w);
        const float2 mh = pdup(-sg * w.z), ml = pdup(-sg * w.w);
        g.re = fma(DF2(rh, rl), hp[b].re, g.re);
        g.re = fma(DF2(mh, ml), hp[b].im, g.re);
        g.im = fma(DF2(rh, rl), hp[b].im, g.im);
        g.im = fma(DF2(ih, il), hp[b].re, g.im);
      }
      up[a].re = up[a].re + g.re;
      up[a].im = up[a].im + g.im;
      auto part = [&](const DF2& v, float f) {
        const float2 m = pmul(pdup(f), sl);
        return DF2{pmul(m, pswap(v.hi, sw)), pmul(m, pswap(v.lo, sw))};
      };
      const DF2 tr = im ? part(g.im, -1.f) : part(g.re, 1.f), ti = im ? part(g.re, 1.f) : part(g.im, 1.f);
      lw[a].re = lw[a].re + tr;
      lw[a].im = lw[a].im + ti;
    }
  }
  // D e = A e - hops / 2; lanes now pair component k with 6 + k
  float2 pr[6], pi[6];
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    const float4 a = __ldg(er + (size_t)j * V + site), b = __ldg(er + (size_t)(3 + j) * V + site);
    pr[2 * j] = make_float2(a.x, b.x);
    pi[2 * j] = make_float2(a.y, b.y);
    pr[2 * j + 1] = make_float2(a.z, b.z);
    pi[2 * j + 1] = make_float2(a.w, b.w);
  }
  const double sc = scale[rhs];
  double2* p = r + (size_t)rhs * 12 * V + site;
  // element k of both packed blocks: two reals per float4
  auto elem = [&](int k, float2& hi, float2& lo) {
    const float4 a = __ldg(C + (size_t)(k / 2) * V + site), b = __ldg(C + (size_t)(18 + k / 2) * V + site);
    hi = k & 1 ? make_float2(a.z, b.z) : make_float2(a.x, b.x);
    lo = k & 1 ? make_float2(a.w, b.w) : make_float2(a.y, b.y);
  };
#pragma unroll
  for (int i = 0; i < 6; ++i) {
    // hops of components i (spins 0, 1) and 6 + i (spins 2, 3)
    const int c = i % 3;
    const bool second = i >= 3;
    auto pick = [&](const DF2& u, const DF2& l) {
      return DF2{pmul(pdup(-0.5f), second ? make_float2(u.hi.y, l.hi.y) : make_float2(u.hi.x, l.hi.x)),
                 pmul(pdup(-0.5f), second ? make_float2(u.lo.y, l.lo.y) : make_float2(u.lo.x, l.lo.x))};
    };
    CD2 o{pick(up[c].re, lw[c].re), pick(up[c].im, lw[c].im)};
    float2 dh, dl;
    elem(i, dh, dl);
    o.re = fma(DF2(dh, dl), pr[i], o.re);
    o.im = fma(DF2(dh, dl), pi[i], o.im);
#pragma unroll
    for (int j = 0; j < 6; ++j) {
      if (j == i) continue;
      const int k = 6 + 2 * (i < j ? offdiag_slot(i, j) : offdiag_slot(j, i));
      float2 rh, rl, ih, il;
      elem(k, rh, rl);
      elem(k + 1, ih, il);
      if (i > j) {  // conjugate element
        ih = pneg(ih);
        il = pneg(il);
      }
      o.re = fma(DF2(rh, rl), pr[j], o.re);
      o.re = fma(DF2(pneg(ih), pneg(il)), pi[j], o.re);
      o.im = fma(DF2(rh, rl), pi[j], o.im);
      o.im = fma(DF2(ih, il), pr[j], o.im);
    }
    bool other = false;
    auto sum = [&](float hi, float lo) { return f2d_fast(hi, other) + f2d_fast(lo, other); };
    double2 d0 = make_double2(sum(o.re.hi.x, o.re.lo.x), sum(o.im.hi.x, o.im.lo.x));
    double2 d1 = make_double2(sum(o.re.hi.y, o.re.lo.y), sum(o.im.hi.y, o.im.lo.y));
    if (other) {
      d0 = make_double2((double)o.re.hi.x + (double)o.re.lo.x, (double)o.im.hi.x + (double)o.im.lo.x);
      d1 = make_double2((double)o.re.hi.y + (double)o.re.lo.y, (double)o.im.hi.y + (double)o.im.lo.y);
    }
    double2 v0 = p[(size_t)i * V], v1 = p[(size_t)(6 + i) * V];
    v0.x -= sc * d0.x;
    v0.y -= sc * d0.y;
    v1.x -= sc * d1.x;
    v1.y -= sc * d1.y;
    p[(size_t)i * V] = v0;
    p[(size_t)(6 + i) * V] = v1;
  }
}

// FP64 values split into double-float pairs, elementwise (two per float4)
__global__ void split_df_kernel(const double2* __restrict__ in, float4* __restrict__ out, size_t n) {
  const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double2 v = in[i];
  const DF a(v.x), b(v.y);
  out[i] = make_float4(a.hi, a.lo, b.hi, b.lo);
}

mglma_status gauge_df_ready(mglma_gauge_s* G, cudaStream_t s) {
  std::lock_guard<std::mutex> lock(G->eo_mu);
  if (G->Udf && G->Cdf) return MGLMA_OK;
  const size_t n = 36 * (size_t)G->g.V;  // link components, pairs of clover reals
  cudaError_t e = cudaMalloc(&G->Udf, n * sizeof(float4));
  if (!e) e = cudaMalloc(&G->Cdf, n * sizeof(float4));
  if (!e) {
    split_df_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(G->U64, G->Udf, n);
    split_df_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(G->C64, G->Cdf, n);
    e = cudaGetLastError();
    if (!e) e = cudaStreamSynchronize(s);  // other streams use them without waiting
    if (!e) return MGLMA_OK;
  }
  cudaGetLastError();
  cudaFree(G->Udf);
  cudaFree(G->Cdf);
  G->Udf = G->Cdf = nullptr;
  if (e == cudaErrorMemoryAllocation)
    return fail(MGLMA_ERR_OOM, "mg solve: no memory for the double-float links and clover");
  MG_CUDA(e);
  return MGLMA_OK;
}

mglma_status dslash_resid_df(mglma_ctx ctx, const mglma_gauge_s* G, const Spinor& e, Spinor& r, const double* scale,
                             cudaStream_t s) {
  if (e.prec != MGLMA_FP32 || r.prec != MGLMA_FP64 || e.V != G->g.V || r.V != G->g.V || e.nrhs != r.nrhs || !scale)
    return fail(MGLMA_ERR_INVALID, "dslash_resid_df: FP32 e, FP64 r of the gauge field's volume and a scale needed");
  if (e.nrhs == 0) return MGLMA_OK;
  MG_CHECK(gauge_df_ready(const_cast<mglma_gauge_s*>(G), s));
  // links and clover as FP64-sized double-float words, e in FP32, r read and written in FP64
  ProfScope ps(ctx, K_DSLASH64, s, (double)e.V * (1152.0 + 480.0 * e.nrhs), 1896.0 * (double)e.V * e.nrhs);
  const size_t ctas = (size_t)((e.V + 127) / 128) * e.nrhs;
  resid_df_kernel<<<(unsigned)ctas, 128, 0, s>>>((const float4*)e.p, (double2*)r.p, G->Udf, G->Cdf,
                                                 make_latidx(G->g.L), (float)G->g.t_bc, e.nrhs, scale);
  MG_LAUNCH_CHECK();
  return MGLMA_OK;
}

}  // namespace mglma
