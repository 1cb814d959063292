// Time-slice contractions of the stochastic estimator (Sec. 5, Eq. C_stoch2)
// and the gamma5 gamma_k sources they need.
//
// For one noise source eta on time slice y0 the estimator of the isovector
// vector correlator between levels i and j is
//   G_ij(x0, y0) = -(1 / (3 L^3)) sum_{k=1}^{3} sum_{x in slice x0}
//                  < (S_j gamma5 gamma_k^dag eta)(x), gamma5 gamma_k (S_i eta)(x) >
// (<u, v> = sum over spin and colour of conj(u) v).  mglma_contract takes the
// solved fields a_k = S_j gamma5 gamma_k^dag eta (k = 1, 2, 3) and
// b = S_i eta and returns G for every x0; mglma_gamma5_gamma makes the
// sources gamma5 gamma_k eta (gamma_k is Hermitian in the chiral basis).
//
// Chiral basis: gamma_k = [[0, -i sigma_k], [i sigma_k, 0]] and
// gamma5 = diag(1, 1, -1, -1), so gamma5 gamma_k = [[0, -i sigma_k],
// [-i sigma_k, 0]]: the upper spin pair of gamma5 gamma_k b is -i sigma_k
// times the lower pair of b, and vice versa.
//
// A CTA takes a chunk of 1024 sites of one (RHS, time slice), a thread one colour
// of a site at a time (four spins of four canonical spinors, so a warp reads
// whole sectors), and sums in FP64 in a fixed order; the chunks of a slice are
// added in order, so results do not depend on timing or on how RHS are batched.
// FP64-pipe bound: 144 FP64 FMAs per site and RHS at about 2 per clock and SM
// against 768 bytes, so every product is one FMA (sums of products let the
// compiler spend three instructions per two).  48x24^3, 12 RHS: 3277 us as one
// CTA per slice with 216 instructions per site.
#include <string>

#include "internal.h"

namespace mglma {

// w = -i sigma_k (u0, u1) for one colour
__device__ __forceinline__ void minus_i_sigma(int k, double2 u0, double2 u1, double2& w0, double2& w1) {
  // -i (x + i y) = y - i x
  auto mi = [](double2 z) { return make_double2(z.y, -z.x); };
  if (k == 1) {  // sigma_1 (u0, u1) = (u1, u0)
    w0 = mi(u1);
    w1 = mi(u0);
  } else if (k == 2) {  // sigma_2 (u0, u1) = (-i u1, i u0); -i sigma_2 = (-u1, u0)
    w0 = make_double2(-u1.x, -u1.y);
    w1 = u0;
  } else {  // sigma_3 (u0, u1) = (u0, -u1)
    w0 = mi(u0);
    w1 = make_double2(-mi(u1).x, -mi(u1).y);
  }
}

constexpr int kChunk = 1024;  // sites per CTA

// part[r][x0][chunk] = sum_k sum_{x in chunk of x0} <a[r][k-1](x), gamma5 gamma_k b[r](x)>,
// times scale, on a grid of (L0 nc, nrhs); on (L0, nrhs) a CTA adds its slice's nc
// chunks in the same order (no room for partial sums, or a stream capture, whose
// graph would own an allocation otherwise: the 48x24^3 case then takes the time of
// one CTA per slice)
__global__ void __launch_bounds__(256) contract_kernel(const double2* __restrict__ a, const double2* __restrict__ b,
                                                       int64_t V, int64_t slice, int nc, int L0, double scale,
                                                       double2* __restrict__ part) {
  const int per = (int)gridDim.x / L0;  // CTAs per slice: nc or 1
  const int x0 = blockIdx.x / per, r = blockIdx.y;
  __shared__ double sh[8][2];
  double2 sum = make_double2(0.0, 0.0);
  for (int chunk = blockIdx.x % per; chunk < nc; chunk += per) {
    const int64_t s0 = (int64_t)chunk * kChunk;
    const int n = 3 * (int)min((int64_t)kChunk, slice - s0);
    const int64_t site0 = (int64_t)x0 * slice + s0;
    double sr = 0.0, si = 0.0;
    for (int t = threadIdx.x; t < n; t += 256) {
      const size_t e = (size_t)(site0 + t / 3) * 12 + t % 3;
      double2 bv[4];
#pragma unroll
      for (int sp = 0; sp < 4; ++sp) bv[sp] = __ldg(b + (size_t)r * V * 12 + e + 3 * sp);
#pragma unroll
      for (int k = 1; k <= 3; ++k) {
        const double2* ak = a + ((size_t)r * 3 + (k - 1)) * V * 12 + e;
        double2 g[4];
        minus_i_sigma(k, bv[2], bv[3], g[0], g[1]);  // upper = -i sigma_k b_lower
        minus_i_sigma(k, bv[0], bv[1], g[2], g[3]);  // lower = -i sigma_k b_upper
#pragma unroll
        for (int sp = 0; sp < 4; ++sp) {
          const double2 u = __ldg(ak + 3 * sp), w = g[sp];
          sr = fma(u.x, w.x, sr);
          sr = fma(u.y, w.y, sr);
          si = fma(u.x, w.y, si);
          si = fma(-u.y, w.x, si);
        }
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      sr += __shfl_down_sync(0xffffffffu, sr, o);
      si += __shfl_down_sync(0xffffffffu, si, o);
    }
    if (threadIdx.x % 32 == 0) {
      sh[threadIdx.x / 32][0] = sr;
      sh[threadIdx.x / 32][1] = si;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      sr = si = 0.0;
      for (int w = 0; w < 8; ++w) {
        sr += sh[w][0];
        si += sh[w][1];
      }
      // product and sum rounded separately, as when contract_sum_kernel adds the
      // chunks: both grids give the same bits
      sum = make_double2(__dadd_rn(sum.x, __dmul_rn(scale, sr)), __dadd_rn(sum.y, __dmul_rn(scale, si)));
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) part[(size_t)r * gridDim.x + blockIdx.x] = sum;
}

// out[i] = sum of the nc chunks of slice i
__global__ void contract_sum_kernel(const double2* __restrict__ part, int nc, int n, double2* __restrict__ out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  double sr = 0.0, si = 0.0;
  for (int c = 0; c < nc; ++c) {
    const double2 v = part[(size_t)i * nc + c];
    sr += v.x;
    si += v.y;
  }
  out[i] = make_double2(sr, si);
}

// out = gamma5 gamma_k in, canonical spinors, one thread per (site, colour)
__global__ void gamma5_gamma_kernel(const double2* __restrict__ in, double2* __restrict__ out, int64_t n, int k) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;  // (rhs * V + site) * 3 + c
  if (t >= n) return;
  const int64_t sv = t / 3;
  const int c = (int)(t % 3);
  const double2* p = in + sv * 12;
  double2* q = out + sv * 12;
  double2 w0, w1, w2, w3;
  minus_i_sigma(k, p[6 + c], p[9 + c], w0, w1);
  minus_i_sigma(k, p[c], p[3 + c], w2, w3);
  q[c] = w0;
  q[3 + c] = w1;
  q[6 + c] = w2;
  q[9 + c] = w3;
}

static mglma_status lattice_volume(const mglma_lattice* lat, int64_t* V, const char* who) {
  *V = 1;
  for (int m = 0; m < 4; ++m) {
    if (lat->L[m] < 1 || lat->L[m] > 4096) return fail(MGLMA_ERR_INVALID, std::string(who) + ": bad extent");
    *V *= lat->L[m];
  }
  return MGLMA_OK;
}

}  // namespace mglma

using namespace mglma;

extern "C" mglma_status mglma_contract(mglma_ctx ctx, const mglma_lattice* lat, int nrhs, const double* a,
                                       const double* b, double* out, void* cuda_stream) {
  if (!ctx || !lat || !a || !b || !out) return fail(MGLMA_ERR_INVALID, "contract: NULL argument");
  if (nrhs < 0) return fail(MGLMA_ERR_INVALID, "contract: nrhs < 0");
  int64_t V = 0;
  MG_CHECK(lattice_volume(lat, &V, "contract"));
  if (nrhs == 0) return MGLMA_OK;
  if (nrhs > 65535) return fail(MGLMA_ERR_INVALID, "contract: at most 65535 RHS per call");
  MG_CUDA(cudaSetDevice(ctx->device));
  cudaStream_t s = pick_stream(ctx, cuda_stream);
  const int64_t slice = V / lat->L[0];
  const size_t bb = (size_t)nrhs * V * 24 * sizeof(double);
  const size_t ob = (size_t)nrhs * lat->L[0] * 2 * sizeof(double);
  Staged ia, ib, o;
  MG_CHECK(stage_in(ctx, a, 3 * bb, s, ia));
  MG_CHECK(stage_in(ctx, b, bb, s, ib));
  MG_CHECK(stage_out_alloc(ctx, out, ob, s, o));
  // one CTA per slice writes the result itself, one per chunk leaves partial sums
  const int nc = (int)((slice + kChunk - 1) / kChunk);
  const int64_t nout = (int64_t)nrhs * lat->L[0], lim = (int64_t)1 << 31;
  double2* part = (double2*)o.dev;
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  if (nc > 1) MG_CUDA(cudaStreamIsCapturing(s, &cap));
  bool split = nc > 1 && cap == cudaStreamCaptureStatusNone && (int64_t)nc * lat->L[0] < lim && nout < lim;
  if (split && dalloc(ctx, (void**)&part, (size_t)nout * nc * sizeof(double2), s) != MGLMA_OK) {
    split = false;
    part = (double2*)o.dev;
  }
  {
    // algorithmic traffic: four spinors per site and RHS read once
    ProfScope ps(ctx, K_CONTRACT, s, 4.0 * (double)bb, 288.0 * (double)V * nrhs);
    contract_kernel<<<dim3((unsigned)((split ? nc : 1) * lat->L[0]), (unsigned)nrhs), 256, 0, s>>>(
        (const double2*)ia.dev, (const double2*)ib.dev, V, slice, nc, lat->L[0], -1.0 / (3.0 * (double)slice), part);
    if (split) contract_sum_kernel<<<(unsigned)((nout + 127) / 128), 128, 0, s>>>(part, nc, (int)nout, (double2*)o.dev);
  }
  const cudaError_t launched = cudaGetLastError();
  if (split) dfree(ctx, part, s);
  MG_CUDA(launched);
  MG_CHECK(stage_out_finish(out, ob, s, o));
  return MGLMA_OK;
}

extern "C" mglma_status mglma_gamma5_gamma(mglma_ctx ctx, const mglma_lattice* lat, int k, int nrhs,
                                           const double* in, double* out, void* cuda_stream) {
  if (!ctx || !lat || !in || !out) return fail(MGLMA_ERR_INVALID, "gamma5_gamma: NULL argument");
  if (k < 1 || k > 3) return fail(MGLMA_ERR_INVALID, "gamma5_gamma: k must be 1, 2 or 3");
  if (nrhs < 0) return fail(MGLMA_ERR_INVALID, "gamma5_gamma: nrhs < 0");
  if (in == out) return fail(MGLMA_ERR_INVALID, "gamma5_gamma: in and out must differ");
  int64_t V = 0;
  MG_CHECK(lattice_volume(lat, &V, "gamma5_gamma"));
  if (nrhs == 0) return MGLMA_OK;
  MG_CUDA(cudaSetDevice(ctx->device));
  cudaStream_t s = pick_stream(ctx, cuda_stream);
  const size_t bytes = (size_t)nrhs * V * 24 * sizeof(double);
  Staged i, o;
  MG_CHECK(stage_in(ctx, in, bytes, s, i));
  MG_CHECK(stage_out_alloc(ctx, out, bytes, s, o));
  const int64_t n = (int64_t)nrhs * V * 3;
  {
    ProfScope ps(ctx, K_PACK, s, 2.0 * (double)bytes);
    gamma5_gamma_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>((const double2*)i.dev, (double2*)o.dev, n, k);
  }
  MG_LAUNCH_CHECK();
  MG_CHECK(stage_out_finish(out, bytes, s, o));
  return MGLMA_OK;
}
