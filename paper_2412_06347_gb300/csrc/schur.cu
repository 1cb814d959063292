// Even-odd (Schur) form of the FP32 Wilson-clover stencil: the operator that
// the multigrid solve's FGCR and its smoother run on when every lattice extent
// is even.
//
// With the sites ordered even then odd, D = [[A_ee, H_eo], [H_oe, A_oo]] (A the
// site-local clover term, H the hops) and
//     S x_e = b_e - H_eo A_oo^-1 b_o,  S = A_ee - H_eo A_oo^-1 H_oe,
//     x_o = A_oo^-1 (b_o - H_oe x_e).
// One application of S costs the arithmetic of one application of D (each site
// is the target of eight hops and one 6x6 pair once) on vectors of half the
// length, and an MR step on S damps about what two steps on D do.  The residual
// of the full system is (b' - S x_e, 0) when x_o follows from x_e.
//
// S runs as two launches of one kernel:
//   odd pass   w_o = A_oo^-1 H_oe x_e
//   even pass  y_e = A_ee x_e - H_eo w_o, with what follows it (residual,
//              dots, a whole MR step) in the epilogue.
// w is FP32; x is FP32, or BF16 for the smoother's fields (FP32 too when asked for).
//
// What bounds it: nothing alone.  ncu on 32x16^3, 16 RHS, odd pass with BF16 in /
// even pass of an MR step: issue slots 46 / 39 %, L1 49 / 46 %, DRAM 27 / 37 %, and
// 4.2 / 5.7 warp cycles per instruction wait on loads; 10 to 16 warps per SM measure
// the same.
// The full-lattice stencil it replaces issued 2717 instructions per site and
// RHS; the odd pass issues 1412.  Complex products run as packed FP32 pairs (one
// FFMA2 does (re, im) with a duplicated link real, so a 3x3 complex product is 18
// packed FMAs plus 6 adds instead of 36 FMAs; duplicating the spinor's reals
// instead measured 1788 against 1180 us), the links are stored as all 18 reals
// with the time-boundary sign applied (no third row to rebuild, no hop factor:
// -1/2 rides on the stored inverse clover and on one packed FMA per component),
// and links and clover are parity-split so a warp reads whole sectors.
// 64x32^3, 16 RHS, us: odd pass BF16 1185 / FP32 1345, even pass MR step 1683,
// dot 1546, FGCR image 1790 (one earlier image; 2301 with three); one MR step on S
// (2868) against 3500 for one on D that damps about half as much.  A whole solve to
// 1e-12, when this form came in: 1507 -> 1102 ms.
//
// Fields of one parity: [rhs][6][Vh] float4 (FP32) or [rhs][3][Vh] uint4
// (BF16), Vh = V / 2, site x at index x >> 1.  A row's address is uniform in
// the warp and the site adds a 32-bit byte offset.  (Tiles of 32 sites, whose
// rows differ by constants, measured slower: 1530 against 1221 us for the
// BF16 odd pass, as a shift by a row of x3 then splits every load.)
#include <mutex>
#include <type_traits>

#include "clover_inverse.cuh"
#include "internal.h"
#include "solver.h"
#include "stencil.cuh"

namespace mglma {

// ------------------------------------------------------------ geometry
struct EoGeo {
  uint32_t L0, L1, L2, Lh;  // Lh = L3 / 2
  uint32_t S0, S1, S2;      // half-lattice strides of x0, x1, x2
  uint32_t Vh;
  uint32_t bpp, b1;  // launch order of the CTAs' site blocks, see EoTile (bpp 0: natural)
};

static EoGeo make_eogeo(const int L[4]) {
  EoGeo g;
  g.L0 = L[0];
  g.L1 = L[1];
  g.L2 = L[2];
  g.Lh = L[3] / 2;
  g.S2 = g.Lh;
  g.S1 = g.S2 * g.L2;
  g.S0 = g.S1 * g.L1;
  g.Vh = g.S0 * g.L0;
  g.bpp = g.b1 = 0;
  return g;
}

// half-lattice index u of parity par: coordinates, and the bit that places
// x3 = 2 xh + odd3
struct EoSite {
  uint32_t x0, x1, x2, xh, odd3;
};
__device__ __forceinline__ EoSite eo_coords(const EoGeo& g, uint32_t u, uint32_t par) {
  EoSite s;
  s.xh = u % g.Lh;
  uint32_t t = u / g.Lh;
  s.x2 = t % g.L2;
  t /= g.L2;
  s.x1 = t % g.L1;
  s.x0 = t / g.L1;
  s.odd3 = (s.x0 + s.x1 + s.x2 + par) & 1u;
  return s;
}
// full-lattice index of half-lattice index u
__device__ __forceinline__ uint32_t eo_full(const EoGeo& g, uint32_t u, uint32_t par) {
  return 2 * u + eo_coords(g, u, par).odd3;
}
// half-lattice index (other parity) of the neighbour one step in +mu / -mu
template <int MU, bool FWD>
__device__ __forceinline__ uint32_t eo_nbr(const EoGeo& g, const EoSite& s, uint32_t u) {
  if (MU == 3) {
    if (FWD) return !s.odd3 ? u : (s.xh + 1 == g.Lh ? u - (g.Lh - 1) : u + 1);
    return s.odd3 ? u : (s.xh == 0 ? u + (g.Lh - 1) : u - 1);
  }
  const uint32_t x = MU == 0 ? s.x0 : (MU == 1 ? s.x1 : s.x2);
  const uint32_t L = MU == 0 ? g.L0 : (MU == 1 ? g.L1 : g.L2);
  const uint32_t S = MU == 0 ? g.S0 : (MU == 1 ? g.S1 : g.S2);
  if (FWD) return x + 1 == L ? u - (L - 1) * S : u + S;
  return x == 0 ? u + (L - 1) * S : u - S;
}

// ------------------------------------------------------------ packed FP32 pairs
__device__ __forceinline__ float2 dup(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
// a + SG b
template <int SG>
__device__ __forceinline__ float2 adds(float2 a, float2 b) {
  return SG > 0 ? add2(a, b) : fma2(b, dup(-1.f), a);
}
// a + SG i b
template <int SG>
__device__ __forceinline__ float2 addi(float2 a, float2 b) {
  return SG > 0 ? make_float2(a.x - b.y, a.y + b.x) : make_float2(a.x + b.y, a.y - b.x);
}

// ------------------------------------------------------------ storage
template <typename T>
__device__ __forceinline__ T ldg_row(const void* b, uint32_t Vh, int j, uint32_t u) {
  return __ldg(reinterpret_cast<const T*>(b) + (size_t)j * Vh + u);
}
template <typename T>
__device__ __forceinline__ T& row(void* b, uint32_t Vh, int j, uint32_t u) {
  return reinterpret_cast<T*>(b)[(size_t)j * Vh + u];
}
__device__ __forceinline__ float2 unpack2(uint32_t u) {
  return make_float2(__uint_as_float(u << 16), __uint_as_float(u & 0xffff0000u));
}
__device__ __forceinline__ uint32_t pack2(float2 a) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(a.x, a.y);
  return *reinterpret_cast<const uint32_t*>(&h);
}
// spinor of twelve (re, im) pairs as loaded; PER bytes per site
template <typename S>
struct Sp;
template <>
struct Sp<float> {
  static constexpr uint32_t PER = 96;
  float4 v[6];
  __device__ __forceinline__ void load(const char* b, uint32_t Vh, uint32_t u) {
#pragma unroll
    for (int j = 0; j < 6; ++j) v[j] = ldg_row<float4>(b, Vh, j, u);
  }
  __device__ __forceinline__ float2 get(int k) const {
    return k & 1 ? make_float2(v[k / 2].z, v[k / 2].w) : make_float2(v[k / 2].x, v[k / 2].y);
  }
  __device__ __forceinline__ static void store(char* b, uint32_t Vh, uint32_t u, const float2 s[12]) {
#pragma unroll
    for (int j = 0; j < 6; ++j)
      row<float4>(b, Vh, j, u) = make_float4(s[2 * j].x, s[2 * j].y, s[2 * j + 1].x, s[2 * j + 1].y);
  }
};
template <>
struct Sp<SpinBf16> {
  static constexpr uint32_t PER = 48;
  uint4 v[3];
  __device__ __forceinline__ void load(const char* b, uint32_t Vh, uint32_t u) {
#pragma unroll
    for (int j = 0; j < 3; ++j) v[j] = ldg_row<uint4>(b, Vh, j, u);
  }
  __device__ __forceinline__ float2 get(int k) const {
    const uint4 q = v[k / 4];
    return unpack2(k % 4 == 0 ? q.x : k % 4 == 1 ? q.y : k % 4 == 2 ? q.z : q.w);
  }
  __device__ __forceinline__ static void store(char* b, uint32_t Vh, uint32_t u, const float2 s[12]) {
#pragma unroll
    for (int j = 0; j < 3; ++j)
      row<uint4>(b, Vh, j, u) =
          make_uint4(pack2(s[4 * j]), pack2(s[4 * j + 1]), pack2(s[4 * j + 2]), pack2(s[4 * j + 3]));
  }
};
// RHS r of a field
template <typename S>
__device__ __forceinline__ const char* rhs_of(const void* f, const EoGeo& g, int r) {
  return reinterpret_cast<const char*>(f) + (size_t)r * Sp<S>::PER * g.Vh;
}
template <typename S>
__device__ __forceinline__ char* rhs_of(void* f, const EoGeo& g, int r) {
  return reinterpret_cast<char*>(f) + (size_t)r * Sp<S>::PER * g.Vh;
}

// ------------------------------------------------------------ hop
// h = upper half of (1 + SG gamma_mu) psi (see stencil.cuh)
template <int MU, int SG>
__device__ __forceinline__ void project2(const float2 p[12], float2 h0[3], float2 h1[3]) {
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    if (MU == 0) {
      h0[c] = adds<-SG>(p[c], p[6 + c]);
      h1[c] = adds<-SG>(p[3 + c], p[9 + c]);
    } else if (MU == 1) {  // i sigma_1 (a, b) = (i b, i a)
      h0[c] = addi<-SG>(p[c], p[9 + c]);
      h1[c] = addi<-SG>(p[3 + c], p[6 + c]);
    } else if (MU == 2) {  // (b, -a)
      h0[c] = adds<-SG>(p[c], p[9 + c]);
      h1[c] = adds<SG>(p[3 + c], p[6 + c]);
    } else {  // (i a, -i b)
      h0[c] = addi<-SG>(p[c], p[6 + c]);
      h1[c] = addi<SG>(p[3 + c], p[9 + c]);
    }
  }
}
// acc += (g, SG e_mu^dag g)
template <int MU, int SG>
__device__ __forceinline__ void reconstruct2(int c, float2 g0, float2 g1, float2 acc[12]) {
  acc[c] = add2(acc[c], g0);
  acc[3 + c] = add2(acc[3 + c], g1);
  if (MU == 0) {
    acc[6 + c] = adds<-SG>(acc[6 + c], g0);
    acc[9 + c] = adds<-SG>(acc[9 + c], g1);
  } else if (MU == 1) {
    acc[6 + c] = addi<SG>(acc[6 + c], g1);
    acc[9 + c] = addi<SG>(acc[9 + c], g0);
  } else if (MU == 2) {
    acc[6 + c] = adds<SG>(acc[6 + c], g1);
    acc[9 + c] = adds<-SG>(acc[9 + c], g0);
  } else {
    acc[6 + c] = addi<SG>(acc[6 + c], g0);
    acc[9 + c] = addi<-SG>(acc[9 + c], g1);
  }
}

// links of one parity and direction: reals 0..15 as four float4 rows, then the
// pair (2, 2) as one float2 row (72 B per site)
struct EoLinks {
  const char* p;  // [par][mu]
};
__device__ __forceinline__ void link_load(const EoLinks& U, uint32_t Vh, int par, int mu, uint32_t n, float2 m[9]) {
  const char* b = U.p + (size_t)(par * 4 + mu) * 72 * Vh;
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const float4 v = ldg_row<float4>(b, Vh, j, n);
    m[2 * j] = make_float2(v.x, v.y);
    m[2 * j + 1] = make_float2(v.z, v.w);
  }
  m[8] = ldg_row<float2>(b + (size_t)64 * Vh, Vh, 0, n);
}

// one hop's operands as loaded: the neighbour's spinor and the link
template <typename SI>
struct HopOps {
  Sp<SI> p;
  float2 m[9];
  template <int MU, bool FWD>
  __device__ __forceinline__ void load(const EoGeo& g, const EoSite& s, uint32_t u, int par, const EoLinks& U,
                                       const char* in) {
    const uint32_t n = eo_nbr<MU, FWD>(g, s, u);
    link_load(U, g.Vh, FWD ? par : 1 - par, MU, FWD ? u : n, m);
    p.load(in, g.Vh, n);
  }
};

// acc += (1 + SG gamma_mu) W in(neighbour), W = U (forward) or U^dag
template <typename SI, int MU, bool FWD>
__device__ __forceinline__ void hop2(const HopOps<SI>& o, float2 acc[12]) {
  constexpr int SG = FWD ? -1 : 1;
  float2 h[6];
  {
    float2 p[12];
#pragma unroll
    for (int k = 0; k < 12; ++k) p[k] = o.p.get(k);
    project2<MU, SG>(p, h, h + 3);
  }
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    float2 e[2], f[2];  // products with the real and the imaginary parts
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      const float2 w = FWD ? o.m[3 * a + b] : o.m[3 * b + a];
      const float2 wr = dup(w.x), wi = dup(w.y);
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        e[k] = b ? fma2(wr, h[3 * k + b], e[k]) : mul2(wr, h[3 * k + b]);
        f[k] = b ? fma2(wi, h[3 * k + b], f[k]) : mul2(wi, h[3 * k + b]);
      }
    }
    float2 q[2];
#pragma unroll
    for (int k = 0; k < 2; ++k) q[k] = FWD ? addi<1>(e[k], f[k]) : addi<-1>(e[k], f[k]);
    reconstruct2<MU, SG>(a, q[0], q[1], acc);
  }
}

// sum over the eight hops (without the factor -1/2); the loads of a hop are
// issued before the arithmetic of the one before it
template <typename SI>
__device__ __forceinline__ void hops2(const EoGeo& g, uint32_t u, int par, const EoLinks& U, const char* in,
                                      float2 acc[12]) {
  const EoSite s = eo_coords(g, u, par);
#pragma unroll
  for (int k = 0; k < 12; ++k) acc[k] = make_float2(0.f, 0.f);
  HopOps<SI> x, y;
  x.template load<0, true>(g, s, u, par, U, in);
  y.template load<0, false>(g, s, u, par, U, in);
  hop2<SI, 0, true>(x, acc);
  x.template load<1, true>(g, s, u, par, U, in);
  hop2<SI, 0, false>(y, acc);
  y.template load<1, false>(g, s, u, par, U, in);
  hop2<SI, 1, true>(x, acc);
  x.template load<2, true>(g, s, u, par, U, in);
  hop2<SI, 1, false>(y, acc);
  y.template load<2, false>(g, s, u, par, U, in);
  hop2<SI, 2, true>(x, acc);
  x.template load<3, true>(g, s, u, par, U, in);
  hop2<SI, 2, false>(y, acc);
  y.template load<3, false>(g, s, u, par, U, in);
  hop2<SI, 3, true>(x, acc);
  hop2<SI, 3, false>(y, acc);
}

// o[6] = packed Hermitian 6x6 block c times x[6]
__device__ __forceinline__ void clover2(const float c[36], const float2* x, float2* o) {
#pragma unroll
  for (int i = 0; i < 6; ++i) {
    float2 e = mul2(dup(c[i]), x[i]), f = make_float2(0.f, 0.f), h = make_float2(0.f, 0.f);
#pragma unroll
    for (int j = 0; j < 6; ++j) {
      if (j == i) continue;
      const int k = 6 + 2 * (i < j ? offdiag_slot(i, j) : offdiag_slot(j, i));
      e = fma2(dup(c[k]), x[j], e);
      if (i < j)
        f = fma2(dup(c[k + 1]), x[j], f);
      else
        h = fma2(dup(c[k + 1]), x[j], h);
    }
    if (i == 0)
      o[i] = addi<1>(e, f);
    else if (i == 5)
      o[i] = addi<-1>(e, h);
    else
      o[i] = addi<1>(e, adds<-1>(f, h));
  }
}
// blocks [chi][9][Vh] float4
__device__ __forceinline__ void clover_load2(const char* C, uint32_t Vh, int chi, uint32_t u, float c[36]) {
  const char* b = C + (size_t)chi * 144 * Vh;
#pragma unroll
  for (int j = 0; j < 9; ++j) {
    const float4 v = ldg_row<float4>(b, Vh, j, u);
    c[4 * j] = v.x;
    c[4 * j + 1] = v.y;
    c[4 * j + 2] = v.z;
    c[4 * j + 3] = v.w;
  }
}

// ------------------------------------------------------------ work split
// A CTA of SCHUR_T threads takes nsub times SCHUR_T consecutive sites of one RHS,
// a site per thread at a time (nsub = 4 on large lattices: fewer CTAs to start
// and fewer partial sums; a function of the volume alone, so a RHS's sums do
// not depend on its batch).  The RHS run fastest in launch order, so the CTAs
// that share a block's links and clover are resident together.  Where the
// planes of fixed (x0, x1) hold whole blocks, the planes are walked in slabs of
// b1 values of x1 (x0 inside a slab), which keeps the three x0 slices a slab
// reads in L2: at 64x32^3 and 16 RHS natural order reads 25 MB per slice
// against an L2 whose halves each serve one die.
constexpr int SCHUR_T = 32;
// resident CTAs the register allocation must allow: 10 to 16 measured the same
// within 5 % for the odd pass; 13 was best or next to best for every pass but
// the FGCR image, whose epilogue spills there (10 or 11 fit it)
template <int EV>
constexpr int schur_ctas() {
  return EV == 5 ? 11 : 13;
}
__host__ __device__ inline uint32_t eo_nsub(uint32_t Vh) { return Vh >= (1u << 18) ? 4 : 1; }
__host__ __device__ inline uint32_t eo_blocks(uint32_t Vh) {
  const uint32_t n = SCHUR_T * eo_nsub(Vh);
  return (Vh + n - 1) / n;
}
struct EoTile {
  int r;
  uint32_t blk;  // block in natural order
  __device__ __forceinline__ EoTile(const EoGeo& g, int nrhs) {
    r = (int)(blockIdx.x % (unsigned)nrhs);
    blk = blockIdx.x / (unsigned)nrhs;
    if (g.bpp) {
      const uint32_t k = blk % g.bpp, q = blk / g.bpp;  // block of its plane, plane in launch order
      const uint32_t per = g.L0 * g.b1, x1 = q / per * g.b1 + q % g.b1, x0 = q % per / g.b1;
      blk = (x0 * g.L1 + x1) * g.bpp + k;
    }
  }
};

// ------------------------------------------------------------ odd pass
// w = A_oo^-1 H_oe x, stored from the inverse blocks times -1/2:
//   SRC 0: w = I hops(in)                   (I = -A^-1 / 2)
//   SRC 1: w = -I (hops(in) + 2 src) = A^-1 (src - H in)
//   SRC 2: w = -2 I src = A^-1 src           (no hops)
template <typename SI, int SRC>
__global__ void __launch_bounds__(SCHUR_T, schur_ctas<-1>())
    schur_odd_kernel(const void* __restrict__ in, const void* __restrict__ src, void* __restrict__ w, EoLinks U,
                     const char* __restrict__ I, EoGeo g, int nrhs, int nsub) {
  const EoTile t(g, nrhs);
  for (int k = 0; k < nsub; ++k) {
    const uint32_t u = (t.blk * nsub + k) * SCHUR_T + threadIdx.x;
    if (u >= g.Vh) return;
    float2 acc[12];
    if (SRC != 2) hops2<SI>(g, u, 1, U, rhs_of<SI>(in, g, t.r), acc);
    if (SRC) {
      Sp<float> q;
      q.load(rhs_of<float>(src, g, t.r), g.Vh, u);
#pragma unroll
      for (int j = 0; j < 12; ++j)
        acc[j] = SRC == 1 ? fma2(q.get(j), dup(-2.f), make_float2(-acc[j].x, -acc[j].y)) : mul2(q.get(j), dup(-2.f));
    }
    float2 o[12];
#pragma unroll
    for (int chi = 0; chi < 2; ++chi) {
      float c[36];
      clover_load2(I, g.Vh, chi, u, c);
      clover2(c, acc + 6 * chi, o + 6 * chi);
    }
    Sp<float>::store(rhs_of<float>(w, g, t.r), g.Vh, u, o);
  }
}

// ------------------------------------------------------------ even pass
enum {
  EV_APPLY,  // out = S x                                            (FP32)
  EV_PREP,  // out = b - H_eo w                                     (FP32)
  EV_RES,   // out = b - S x                                        (FP32 b; out SM)
  EV_DOT,   // out = S x, partials of |out|^2 and <out, x>          (SM x, out)
  EV_MR,    // one MR step: with u = S x (x = t_k): out = t_k - a u, sn = s - a t_k,
            // partials of |out|^2 and <out, sn>                     (SM)
  EV_GCR    // out = S x with the FGCR dots                         (FP32)
};
struct EvArgs {
  const void* b = nullptr;
  const void* s = nullptr;
  void* sn = nullptr;
  const float2* alpha = nullptr;
  double* part = nullptr;    // EV_DOT / EV_MR: [rhs][block][3]; EV_GCR: [rhs][block][6]
  const char* W0 = nullptr;  // EV_GCR: earlier images, wslot bytes apart; k of them (k = 0: r)
  size_t wslot = 0;
  int k = 0;
  const void* r = nullptr;
};

// per-thread sums of one site each added over the CTA's warp in FP32 (the FP64 pipe
// of GB300 is too narrow for a per-thread FP64 tree); FP32 never carries more than
// the 32 sites of a warp, whatever nsub is.  The values are halved between the
// lanes while there are several (six values: 9 shuffles instead of 30), so a lane
// ends with the total of value warp_value(lane)
template <int NV>
__device__ __forceinline__ float warp_total(const float (&v)[NV]) {
  static_assert(SCHUR_T == 32 && NV <= 8, "one warp per CTA");
  constexpr int P = NV <= 4 ? 4 : 8;
  float a[P];
#pragma unroll
  for (int i = 0; i < P; ++i) a[i] = i < NV ? v[i < NV ? i : 0] : 0.f;
  int o = 16;
#pragma unroll
  for (int n = P; n > 1; n /= 2, o /= 2) {
    const bool up = threadIdx.x & o;
#pragma unroll
    for (int i = 0; i < n / 2; ++i) {
      const float keep = up ? a[i + n / 2] : a[i], send = up ? a[i] : a[i + n / 2];
      a[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
    }
  }
#pragma unroll
  for (int q = 16 / P; q > 0; q /= 2) a[0] += __shfl_xor_sync(0xffffffffu, a[0], q);
  return a[0];
}
// the value whose total a lane holds; the first lane of each group of 32 / P writes
template <int NV>
__device__ __forceinline__ int warp_value(int lane) {
  return lane / (NV <= 4 ? 8 : 4);
}

// SM: storage of the smoother's fields, SpinBf16 or float
template <int EV, typename SM = SpinBf16>
__global__ void __launch_bounds__(SCHUR_T, schur_ctas<EV>())
    schur_even_kernel(const void* __restrict__ w, const void* __restrict__ x, void* __restrict__ out, EoLinks U,
                      const char* __restrict__ C, EoGeo g, int nrhs, int nsub, EvArgs a) {
  constexpr bool RED = EV == EV_DOT || EV == EV_MR || EV == EV_GCR;
  constexpr int NV = EV == EV_GCR ? 6 : 3;
  constexpr bool BF = std::is_same<SM, SpinBf16>::value;
  using SX = typename std::conditional<EV == EV_DOT || EV == EV_MR, SM, float>::type;
  const EoTile t(g, nrhs);
  const int r = t.r;
  double sum = 0.0;  // of value warp_value(lane)
  for (int k = 0; k < nsub; ++k) {
    const uint32_t u0 = (t.blk * nsub + k) * SCHUR_T, u = u0 + threadIdx.x;
    if (RED ? u0 >= g.Vh : u >= g.Vh) break;
    float v[NV];
#pragma unroll
    for (int e = 0; e < NV; ++e) v[e] = 0.f;
    if (!RED || u < g.Vh) {
      float2 acc[12];
      hops2<float>(g, u, 0, U, rhs_of<float>(w, g, r), acc);
      if (EV == EV_PREP) {
        Sp<float> q;
        q.load(rhs_of<float>(a.b, g, r), g.Vh, u);
#pragma unroll
        for (int j = 0; j < 12; ++j) acc[j] = fma2(acc[j], dup(0.5f), q.get(j));
      } else {  // S x = A x + hops / 2
        Sp<SX> q;
        q.load(rhs_of<SX>(x, g, r), g.Vh, u);
        float2 p[12];
#pragma unroll
        for (int j = 0; j < 12; ++j) p[j] = q.get(j);
#pragma unroll
        for (int chi = 0; chi < 2; ++chi) {
          float c[36];
          float2 o[6];
          clover_load2(C, g.Vh, chi, u, c);
          clover2(c, p + 6 * chi, o);
#pragma unroll
          for (int j = 0; j < 6; ++j) acc[6 * chi + j] = fma2(acc[6 * chi + j], dup(0.5f), o[j]);
        }
      }
      if (EV == EV_PREP || EV == EV_APPLY) {
        Sp<float>::store(rhs_of<float>(out, g, r), g.Vh, u, acc);
      } else if (EV == EV_RES) {
        Sp<float> q;
        q.load(rhs_of<float>(a.b, g, r), g.Vh, u);
#pragma unroll
        for (int j = 0; j < 12; ++j) acc[j] = adds<-1>(q.get(j), acc[j]);
        Sp<SM>::store(rhs_of<SM>(out, g, r), g.Vh, u, acc);
      } else if (EV == EV_DOT) {
        Sp<SM> p;
        p.load(rhs_of<SM>(x, g, r), g.Vh, u);
#pragma unroll
        for (int j = 0; j < 12; ++j) {
          const float2 q = BF ? unpack2(pack2(acc[j])) : acc[j], y = p.get(j);  // the dots see the values as stored
          acc[j] = q;
          v[0] += q.x * q.x + q.y * q.y;
          v[1] += q.x * y.x + q.y * y.y;
          v[2] += q.x * y.y - q.y * y.x;
        }
        Sp<SM>::store(rhs_of<SM>(out, g, r), g.Vh, u, acc);
      } else if (EV == EV_MR) {
        const float2 al = a.alpha[r];
        // complex -a v = nr (re, im) + ni (im, re) with ni = (Im a, -Im a)
        const float2 nr = dup(-al.x), ni = make_float2(al.y, -al.y);
        const char *tp = rhs_of<SM>(x, g, r), *sp = rhs_of<SM>(a.s, g, r);
        char *op = rhs_of<SM>(out, g, r), *np = rhs_of<SM>(a.sn, g, r);
        if constexpr (BF) {
#pragma unroll
          for (int j = 0; j < 3; ++j) {
            const uint4 tv = ldg_row<uint4>(tp, g.Vh, j, u), sv = ldg_row<uint4>(sp, g.Vh, j, u);
            const uint32_t tw[4] = {tv.x, tv.y, tv.z, tv.w}, sw[4] = {sv.x, sv.y, sv.z, sv.w};
            uint32_t to[4], so[4];
#pragma unroll
            for (int h = 0; h < 4; ++h) {
              const float2 tk = unpack2(tw[h]), sk = unpack2(sw[h]), q = acc[4 * j + h];
              to[h] = pack2(fma2(ni, make_float2(q.y, q.x), fma2(nr, q, tk)));
              so[h] = pack2(fma2(ni, make_float2(tk.y, tk.x), fma2(nr, tk, sk)));
              const float2 tn = unpack2(to[h]), sn = unpack2(so[h]);
              v[0] += tn.x * tn.x + tn.y * tn.y;
              v[1] += tn.x * sn.x + tn.y * sn.y;
              v[2] += tn.x * sn.y - tn.y * sn.x;
            }
            row<uint4>(op, g.Vh, j, u) = make_uint4(to[0], to[1], to[2], to[3]);
            row<uint4>(np, g.Vh, j, u) = make_uint4(so[0], so[1], so[2], so[3]);
          }
        } else {
#pragma unroll
          for (int j = 0; j < 6; ++j) {
            const float4 tv = ldg_row<float4>(tp, g.Vh, j, u), sv = ldg_row<float4>(sp, g.Vh, j, u);
            const float2 tk[2] = {make_float2(tv.x, tv.y), make_float2(tv.z, tv.w)};
            const float2 sk[2] = {make_float2(sv.x, sv.y), make_float2(sv.z, sv.w)};
            float2 tn[2], sn[2];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              const float2 q = acc[2 * j + h];
              tn[h] = fma2(ni, make_float2(q.y, q.x), fma2(nr, q, tk[h]));
              sn[h] = fma2(ni, make_float2(tk[h].y, tk[h].x), fma2(nr, tk[h], sk[h]));
              v[0] += tn[h].x * tn[h].x + tn[h].y * tn[h].y;
              v[1] += tn[h].x * sn[h].x + tn[h].y * sn[h].y;
              v[2] += tn[h].x * sn[h].y - tn[h].y * sn[h].x;
            }
            row<float4>(op, g.Vh, j, u) = make_float4(tn[0].x, tn[0].y, tn[1].x, tn[1].y);
            row<float4>(np, g.Vh, j, u) = make_float4(sn[0].x, sn[0].y, sn[1].x, sn[1].y);
          }
        }
      } else {
        Sp<float>::store(rhs_of<float>(out, g, r), g.Vh, u, acc);
        if (a.k == 0) {
          const char* rp = rhs_of<float>(a.r, g, r);
#pragma unroll
          for (int c = 0; c < 6; ++c) {
            const float4 q = ldg_row<float4>(rp, g.Vh, c, u);
            const float2 w0 = acc[2 * c], w1 = acc[2 * c + 1];
            v[0] += w0.x * w0.x + w0.y * w0.y + w1.x * w1.x + w1.y * w1.y;
            v[1] += w0.x * q.x + w0.y * q.y + w1.x * q.z + w1.y * q.w;
            v[2] += w0.x * q.y - w0.y * q.x + w1.x * q.w - w1.y * q.z;
          }
        } else {
#pragma unroll
          for (int j = 0; j < 3; ++j) {
            if (j >= a.k) break;
            const char* wp = rhs_of<float>((const void*)(a.W0 + j * a.wslot), g, r);
#pragma unroll
            for (int c = 0; c < 6; ++c) {
              const float4 q = ldg_row<float4>(wp, g.Vh, c, u);
              const float2 w0 = acc[2 * c], w1 = acc[2 * c + 1];
              v[(2 * j) % NV] += q.x * w0.x + q.y * w0.y + q.z * w1.x + q.w * w1.y;
              v[(2 * j + 1) % NV] += q.x * w0.y - q.y * w0.x + q.z * w1.y - q.w * w1.x;
            }
          }
        }
      }
    }
    if (RED) {
      __syncwarp();
      sum += (double)warp_total(v);
    }
  }
  if (RED) {
    const int e = warp_value<NV>(threadIdx.x);
    if (threadIdx.x % (NV <= 4 ? 8 : 4) == 0 && e < NV)
      a.part[((size_t)r * eo_blocks(g.Vh) + t.blk) * NV + e] = sum;
  }
}

// the MR step's partials of RHS blockIdx.x in a fixed order, then its step
// length alpha = <t, s> / |t|^2
__global__ void __launch_bounds__(512) mr_finish_kernel(const double* __restrict__ part, uint32_t nblk,
                                                        float2* __restrict__ alpha) {
  const int r = blockIdx.x;
  double a = 0, b = 0, c = 0;
  const double* p = part + (size_t)r * nblk * 3;
  for (uint32_t i = threadIdx.x; i < nblk; i += 512) {
    a += p[3 * (size_t)i];
    b += p[3 * (size_t)i + 1];
    c += p[3 * (size_t)i + 2];
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    a += __shfl_down_sync(0xffffffffu, a, o);
    b += __shfl_down_sync(0xffffffffu, b, o);
    c += __shfl_down_sync(0xffffffffu, c, o);
  }
  __shared__ double sh[16][3];
  if (threadIdx.x % 32 == 0) {
    sh[threadIdx.x / 32][0] = a;
    sh[threadIdx.x / 32][1] = b;
    sh[threadIdx.x / 32][2] = c;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    a = b = c = 0;
    for (int w = 0; w < 16; ++w) {
      a += sh[w][0];
      b += sh[w][1];
      c += sh[w][2];
    }
    alpha[r] = a > 0 ? make_float2((float)(b / a), (float)(c / a)) : make_float2(0.f, 0.f);
  }
}

// z += sum_{k<ns} alpha_k s_k (s_k at s + k sstride 16-byte pieces, alpha_k[rhs] at
// alpha + k nrhs): the smoothing steps' iterate, formed once per group of steps, so
// a step moves 288 B per site and RHS instead of 480 (BF16 s_k).  One thread per
// site and group of four components
template <int NS, typename SM>
__global__ void __launch_bounds__(256) mr_iterate_kernel(float4* __restrict__ z, const uint4* __restrict__ s,
                                                         size_t sstride, const float2* __restrict__ alpha, int nrhs,
                                                         uint32_t Vh) {
  constexpr bool BF = std::is_same<SM, SpinBf16>::value;
  constexpr int PIECES = BF ? 1 : 2;  // per group of four components
  const int r = blockIdx.y;
  const uint32_t j = blockIdx.z, u = blockIdx.x * 256 + threadIdx.x;
  if (u >= Vh) return;
  const uint4* sp = s + ((size_t)r * 3 + j) * PIECES * Vh + u;
  float4* z0 = z + ((size_t)r * 6 + 2 * j) * Vh + u;
  uint4 sv[NS][PIECES];
#pragma unroll
  for (int k = 0; k < NS; ++k)
#pragma unroll
    for (int p = 0; p < PIECES; ++p) sv[k][p] = __ldg(sp + k * sstride + (size_t)p * Vh);
  const float4 a = z0[0], c = z0[Vh];
  float2 q[4] = {make_float2(a.x, a.y), make_float2(a.z, a.w), make_float2(c.x, c.y), make_float2(c.z, c.w)};
#pragma unroll
  for (int k = 0; k < NS; ++k) {
    const float2 al = alpha[(size_t)k * nrhs + r];
    const float2 ar = dup(al.x), ai = make_float2(-al.y, al.y);
#pragma unroll
    for (int h = 0; h < 4; ++h) {
      float2 v;
      if constexpr (BF) {
        const uint32_t w[4] = {sv[k][0].x, sv[k][0].y, sv[k][0].z, sv[k][0].w};
        v = unpack2(w[h]);
      } else {
        const uint4 w = sv[k][h / 2];
        v = h % 2 ? make_float2(__uint_as_float(w.z), __uint_as_float(w.w))
                  : make_float2(__uint_as_float(w.x), __uint_as_float(w.y));
      }
      q[h] = fma2(ai, make_float2(v.y, v.x), fma2(ar, v, q[h]));
    }
  }
  z0[0] = make_float4(q[0].x, q[0].y, q[1].x, q[1].y);
  z0[Vh] = make_float4(q[2].x, q[2].y, q[3].x, q[3].y);
}

// ------------------------------------------------------------ set-up copies
// links of parity blockIdx.y: the FP64 links rounded once, all 18 reals, the
// hop across the time boundary multiplied by its sign
__global__ void eo_links_kernel(const double2* __restrict__ U64, char* __restrict__ dst, EoGeo g, float bc) {
  const uint32_t u = blockIdx.x * blockDim.x + threadIdx.x;
  const int par = blockIdx.y / 4, mu = blockIdx.y % 4;
  if (u >= g.Vh) return;
  const EoSite s = eo_coords(g, u, par);
  const uint32_t site = 2 * u + s.odd3;
  const float f = mu == 0 && s.x0 == g.L0 - 1 ? bc : 1.f;
  float2 m[9];
#pragma unroll
  for (int k = 0; k < 9; ++k) {
    const double2 v = U64[((size_t)mu * 9 + k) * 2 * g.Vh + site];
    m[k] = make_float2(f * (float)v.x, f * (float)v.y);
  }
  char* p = dst + (size_t)(par * 4 + mu) * 72 * g.Vh;
#pragma unroll
  for (int j = 0; j < 4; ++j)
    row<float4>(p, g.Vh, j, u) = make_float4(m[2 * j].x, m[2 * j].y, m[2 * j + 1].x, m[2 * j + 1].y);
  row<float2>(p + (size_t)64 * g.Vh, g.Vh, 0, u) = m[8];
}

// clover blocks of the even sites (FP32 of the FP64 blocks), and -1/2 times the
// inverse blocks of the odd sites (inverted in FP64); chirality blockIdx.y.
// *bad is set when a block is singular or an inverse entry is beyond 100 (the
// blocks are of order 4: the caller then keeps the full-lattice operator)
__global__ void __launch_bounds__(128) eo_clover_copy_kernel(const double2* __restrict__ C64, char* __restrict__ Ce,
                                                             char* __restrict__ Io, EoGeo g, int* bad) {
  const uint32_t u = blockIdx.x * blockDim.x + threadIdx.x;
  const int chi = blockIdx.y;
  if (u >= g.Vh) return;
  const int64_t V = 2 * (int64_t)g.Vh;
  double c[36], ci[36];
  Clover<double>::load(C64, V, chi, eo_full(g, u, 0), c);
  char *pe = Ce + (size_t)chi * 144 * g.Vh, *po = Io + (size_t)chi * 144 * g.Vh;
#pragma unroll
  for (int j = 0; j < 9; ++j)
    row<float4>(pe, g.Vh, j, u) = make_float4((float)c[4 * j], (float)c[4 * j + 1], (float)c[4 * j + 2], (float)c[4 * j + 3]);
  Clover<double>::load(C64, V, chi, eo_full(g, u, 1), c);
  bool ok = clover_inverse6(c, ci);
#pragma unroll
  for (int j = 0; j < 36; ++j) {
    ok = ok && fabs(ci[j]) < 100.0;
    ci[j] *= -0.5;
  }
#pragma unroll
  for (int j = 0; j < 9; ++j)
    row<float4>(po, g.Vh, j, u) =
        make_float4((float)ci[4 * j], (float)ci[4 * j + 1], (float)ci[4 * j + 2], (float)ci[4 * j + 3]);
  if (!ok) atomicExch(bad, 1);
}

// ------------------------------------------------------------ full <-> half fields
// FP64 full field times scale[rhs] -> FP32 halves
__global__ void eo_split_kernel(const double2* __restrict__ f, float4* __restrict__ e, float4* __restrict__ o, EoGeo g,
                                const double* __restrict__ scale) {
  const uint32_t u = blockIdx.x * blockDim.x + threadIdx.x;
  const int r = blockIdx.y;
  if (u >= g.Vh) return;
  const double sc = scale[r];
  const uint32_t odd3 = eo_coords(g, u, 0).odd3;
  const size_t V = 2 * (size_t)g.Vh;
  const double2* p = f + (size_t)r * 12 * V + 2 * (size_t)u;
#pragma unroll
  for (int par = 0; par < 2; ++par) {
    float4* d = (par ? o : e) + (size_t)r * 6 * g.Vh + u;
    const double2* q = p + (odd3 ^ (uint32_t)par);
#pragma unroll
    for (int j = 0; j < 6; ++j) {
      const double2 a = q[(size_t)(2 * j) * V], b = q[(size_t)(2 * j + 1) * V];
      d[(size_t)j * g.Vh] =
          make_float4((float)(sc * a.x), (float)(sc * a.y), (float)(sc * b.x), (float)(sc * b.y));
    }
  }
}

// FP32 halves -> FP32 full field f, and x (FP64 full) += scale[rhs] f
__global__ void eo_join_kernel(const float4* __restrict__ e, const float4* __restrict__ o, float4* __restrict__ f,
                               double2* __restrict__ x, EoGeo g, const double* __restrict__ scale) {
  const uint32_t u = blockIdx.x * blockDim.x + threadIdx.x;
  const int r = blockIdx.y;
  if (u >= g.Vh) return;
  const double sc = scale[r];
  const uint32_t odd3 = eo_coords(g, u, 0).odd3;
  const size_t V = 2 * (size_t)g.Vh;
#pragma unroll
  for (int j = 0; j < 6; ++j) {
    const size_t h = ((size_t)r * 6 + j) * g.Vh + u;
    const float4 v[2] = {e[h], o[h]};
#pragma unroll
    for (int par = 0; par < 2; ++par) {
      const size_t site = 2 * (size_t)u + (odd3 ^ (uint32_t)par);
      f[((size_t)r * 6 + j) * V + site] = v[par];
      double2* a = x + ((size_t)r * 12 + 2 * j) * V + site;
      a[0] = make_double2(a[0].x + sc * (double)v[par].x, a[0].y + sc * (double)v[par].y);
      a[V] = make_double2(a[V].x + sc * (double)v[par].z, a[V].y + sc * (double)v[par].w);
    }
  }
}

// FP32 even half -> full field, zero on the odd sites; and back (even sites)
__global__ void eo_embed_kernel(const float4* __restrict__ e, float4* __restrict__ f, EoGeo g) {
  const uint32_t u = blockIdx.x * blockDim.x + threadIdx.x;
  const int r = blockIdx.y;
  if (u >= g.Vh) return;
  const uint32_t odd3 = eo_coords(g, u, 0).odd3;
  const size_t V = 2 * (size_t)g.Vh;
#pragma unroll
  for (int j = 0; j < 6; ++j) {
    float4* d = f + ((size_t)r * 6 + j) * V + 2 * (size_t)u;
    d[odd3] = e[((size_t)r * 6 + j) * g.Vh + u];
    d[odd3 ^ 1u] = make_float4(0.f, 0.f, 0.f, 0.f);
  }
}
__global__ void eo_extract_kernel(const float4* __restrict__ f, float4* __restrict__ e, EoGeo g) {
  const uint32_t u = blockIdx.x * blockDim.x + threadIdx.x;
  const int r = blockIdx.y;
  if (u >= g.Vh) return;
  const uint32_t odd3 = eo_coords(g, u, 0).odd3;
  const size_t V = 2 * (size_t)g.Vh;
#pragma unroll
  for (int j = 0; j < 6; ++j)
    e[((size_t)r * 6 + j) * g.Vh + u] = f[((size_t)r * 6 + j) * V + 2 * (size_t)u + odd3];
}

// ============================================================ host side
// fine_eo_ready with eo_mu held
static mglma_status form_copies(mglma_ctx ctx, mglma_gauge_s* G, bool* usable, cudaStream_t s) {
  *usable = false;
  if (G->eo_state < 0) return MGLMA_OK;
  if (G->eo_state > 0) {
    *usable = true;
    return MGLMA_OK;
  }
  for (int m = 0; m < 4; ++m)
    if (G->g.L[m] % 2) {
      G->eo_state = -1;
      return MGLMA_OK;
    }
  if (G->g.V >= (int64_t)1 << 31) {  // 32-bit site indices
    G->eo_state = -1;
    return MGLMA_OK;
  }
  const EoGeo g = make_eogeo(G->g.L);
  const size_t Vh = g.Vh;
  int* bad = nullptr;
  cudaError_t e = cudaMalloc(&G->Ueo, Vh * 8 * 72);
  if (!e) e = cudaMalloc(&G->Ceo, Vh * 288);
  if (!e) e = cudaMalloc(&G->Ieo, Vh * 288);
  if (!e) e = cudaMalloc(&bad, sizeof(int));
  int h = 0;
  if (!e) {
    ProfScope ps(ctx, K_SETUP, s);
    cudaMemsetAsync(bad, 0, sizeof(int), s);
    eo_links_kernel<<<dim3((unsigned)((Vh + 127) / 128), 8), 128, 0, s>>>(G->U64, G->Ueo, g, (float)G->g.t_bc);
    eo_clover_copy_kernel<<<dim3((unsigned)((Vh + 127) / 128), 2), 128, 0, s>>>(G->C64, G->Ceo, G->Ieo, g, bad);
    e = cudaGetLastError();
    if (!e) e = cudaMemcpyAsync(&h, bad, sizeof(int), cudaMemcpyDeviceToHost, s);
    if (!e) e = cudaStreamSynchronize(s);
  }
  cudaFree(bad);
  if (!e && !h) {
    G->eo_state = 1;
    *usable = true;
    return MGLMA_OK;
  }
  // no memory for the copies, or a block that cannot be inverted well: the
  // full-lattice operator serves
  cudaFree(G->Ueo);
  cudaFree(G->Ceo);
  cudaFree(G->Ieo);
  G->Ueo = G->Ceo = G->Ieo = nullptr;
  if (h) G->eo_state = -1;
  if (e == cudaErrorMemoryAllocation) {
    cudaGetLastError();
    return MGLMA_OK;
  }
  MG_CUDA(e);
  return MGLMA_OK;
}

mglma_status fine_eo_ready(mglma_ctx ctx, mglma_gauge_s* G, bool* usable, cudaStream_t s) {
  std::lock_guard<std::mutex> lock(G->eo_mu);
  return form_copies(ctx, G, usable, s);
}

mglma_status EoUse::acquire(mglma_ctx ctx, const mglma_gauge_s* g, cudaStream_t s) {
  mglma_gauge_s* gg = const_cast<mglma_gauge_s*>(g);
  std::lock_guard<std::mutex> lock(gg->eo_mu);
  MG_CHECK(form_copies(ctx, gg, &usable, s));
  if (usable) {
    G = gg;
    ++G->eo_users;
  }
  return MGLMA_OK;
}

void EoUse::release(bool free) {
  if (!G) return;
  std::lock_guard<std::mutex> lock(G->eo_mu);
  if (--G->eo_users == 0 && free) {
    cudaFree(G->Ueo);
    cudaFree(G->Ceo);
    cudaFree(G->Ieo);
    G->Ueo = G->Ceo = G->Ieo = nullptr;
    G->eo_state = 0;
  }
  G = nullptr;
  usable = false;
}

static EoLinks eo_links(const mglma_gauge_s* G) { return EoLinks{G->Ueo}; }
static unsigned schur_blocks(const mglma_gauge_s* G) { return eo_blocks((uint32_t)(G->g.V / 2)); }

static mglma_status eo_shape(const mglma_gauge_s* G, std::initializer_list<const Spinor*> f, const char* who) {
  if (G->eo_state <= 0) return fail(MGLMA_ERR_INVALID, std::string(who) + ": even-odd copies missing");
  for (const Spinor* v : f)
    if (v->V != G->g.V / 2 || v->nrhs != (*f.begin())->nrhs)
      return fail(MGLMA_ERR_INVALID, std::string(who) + ": half-lattice fields of one RHS count needed");
  return MGLMA_OK;
}

// with the launch order of nrhs RHS (see EoTile): the widest slab whose three
// slices stay within 32 MB (64x32^3, 16 RHS, average of the passes: natural
// order 1740 us, 64 / 32 / 16 / 8 MB 1679 / 1651 / 1661 / 1699 us)
static EoGeo launch_geo(const mglma_gauge_s* G, int nrhs) {
  EoGeo g = make_eogeo(G->g.L);
  const uint32_t plane = g.S1, blk = SCHUR_T * eo_nsub(g.Vh);
  if (plane % blk) return g;
  uint32_t b1 = g.L1;
  while (b1 > 1 && (g.L1 % b1 || 3.0 * b1 * plane * 96.0 * nrhs > 32e6)) --b1;
  if (b1 == g.L1) return g;
  g.bpp = plane / blk;
  g.b1 = b1;
  return g;
}

template <typename SI, int SRC>
static void launch_odd(const mglma_gauge_s* G, const Spinor* in, const Spinor* src, Spinor& w, cudaStream_t s) {
  schur_odd_kernel<SI, SRC><<<schur_blocks(G) * (unsigned)w.nrhs, SCHUR_T, 0, s>>>(
      in ? in->p : nullptr, src ? src->p : nullptr, w.p, eo_links(G), G->Ieo, launch_geo(G, w.nrhs), w.nrhs,
      (int)eo_nsub((uint32_t)(G->g.V / 2)));
}

// algorithmic bytes of a pass: links (288 B per site of the lattice) and one
// parity's clover blocks once, the fields as given per half-lattice site and RHS
static double schur_bytes(const mglma_gauge_s* G, int nrhs, double per_site) {
  const double Vh = 0.5 * (double)G->g.V;
  return Vh * (576.0 + 288.0 + per_site * nrhs);
}
static double schur_flops(const mglma_gauge_s* G, int nrhs) { return 0.5 * 1896.0 * (double)G->g.V * nrhs; }

mglma_status schur_odd(mglma_ctx ctx, const mglma_gauge_s* G, const Spinor& in, Spinor& w, cudaStream_t s) {
  MG_CHECK(eo_shape(G, {&w, &in}, "schur_odd"));
  if (w.nrhs == 0) return MGLMA_OK;
  const bool bf = in.prec == MGLMA_BF16;
  ProfScope ps(ctx, K_DSLASH32, s, schur_bytes(G, w.nrhs, bf ? 144.0 : 192.0), schur_flops(G, w.nrhs));
  if (bf)
    launch_odd<SpinBf16, 0>(G, &in, nullptr, w, s);
  else
    launch_odd<float, 0>(G, &in, nullptr, w, s);
  MG_LAUNCH_CHECK();
  return MGLMA_OK;
}

mglma_status schur_odd_solution(mglma_ctx ctx, const mglma_gauge_s* G, const Spinor* xe, const Spinor& bo, Spinor& xo,
                                cudaStream_t s) {
  MG_CHECK(eo_shape(G, {&xo, &bo, xe ? xe : &bo}, "schur_odd_solution"));
  if (xo.nrhs == 0) return MGLMA_OK;
  ProfScope ps(ctx, K_DSLASH32, s, schur_bytes(G, xo.nrhs, 288.0), schur_flops(G, xo.nrhs));
  if (xe)
    launch_odd<float, 1>(G, xe, &bo, xo, s);
  else
    launch_odd<float, 2>(G, nullptr, &bo, xo, s);
  MG_LAUNCH_CHECK();
  return MGLMA_OK;
}

template <int EV, typename SM = SpinBf16>
static void launch_even(const mglma_gauge_s* G, const Spinor& w, const void* x, void* out, const EvArgs& a,
                        cudaStream_t s) {
  schur_even_kernel<EV, SM><<<schur_blocks(G) * (unsigned)w.nrhs, SCHUR_T, 0, s>>>(
      w.p, x, out, eo_links(G), G->Ceo, launch_geo(G, w.nrhs), w.nrhs, (int)eo_nsub((uint32_t)(G->g.V / 2)), a);
}

mglma_status schur_prepare(mglma_ctx ctx, const mglma_gauge_s* G, const Spinor& be, const Spinor& vo, Spinor& out,
                           cudaStream_t s) {
  MG_CHECK(eo_shape(G, {&out, &be, &vo}, "schur_prepare"));
  if (out.nrhs == 0) return MGLMA_OK;
  EvArgs a;
  a.b = be.p;
  ProfScope ps(ctx, K_DSLASH32, s, schur_bytes(G, out.nrhs, 288.0), schur_flops(G, out.nrhs));
  launch_even<EV_PREP>(G, vo, nullptr, out.p, a, s);
  MG_LAUNCH_CHECK();
  return MGLMA_OK;
}

mglma_status schur_apply(mglma_ctx ctx, const mglma_gauge_s* G, const Spinor& w, const Spinor& x, Spinor& out,
                         cudaStream_t s) {
  MG_CHECK(eo_shape(G, {&out, &w, &x}, "schur_apply"));
  if (out.nrhs == 0) return MGLMA_OK;
  ProfScope ps(ctx, K_DSLASH32, s, schur_bytes(G, out.nrhs, 288.0), schur_flops(G, out.nrhs));
  launch_even<EV_APPLY>(G, w, x.p, out.p, EvArgs(), s);
  MG_LAUNCH_CHECK();
  return MGLMA_OK;
}

mglma_status schur_resid(mglma_ctx ctx, const mglma_gauge_s* G, const Spinor& w, const Spinor& x, const Spinor& b,
                         Spinor& out, cudaStream_t s) {
  MG_CHECK(eo_shape(G, {&out, &w, &x, &b}, "schur_resid"));
  if (out.nrhs == 0) return MGLMA_OK;
  EvArgs a;
  a.b = b.p;
  const bool bf = out.prec == MGLMA_BF16;
  ProfScope ps(ctx, K_DSLASH32, s, schur_bytes(G, out.nrhs, bf ? 336.0 : 384.0), schur_flops(G, out.nrhs));
  if (bf)
    launch_even<EV_RES>(G, w, x.p, out.p, a, s);
  else
    launch_even<EV_RES, float>(G, w, x.p, out.p, a, s);
  MG_LAUNCH_CHECK();
  return MGLMA_OK;
}

size_t schur_part_doubles(int64_t V, int nrhs) { return (size_t)6 * nrhs * eo_blocks((uint32_t)(V / 2)); }

static mglma_status mr_finish(mglma_ctx ctx, const mglma_gauge_s* G, const double* part, int nrhs, float2* alpha,
                              cudaStream_t s) {
  const uint32_t nblk = schur_blocks(G);
  ProfScope ps(ctx, K_REDUCE, s, 24.0 * nblk * nrhs);
  mr_finish_kernel<<<nrhs, 512, 0, s>>>(part, nblk, alpha);
  MG_LAUNCH_CHECK();
  return MGLMA_OK;
}

mglma_status schur_dot(mglma_ctx ctx, const mglma_gauge_s* G, const Spinor& w, const Spinor& x, Spinor& out,
                       double* part, float2* alpha, cudaStream_t s) {
  MG_CHECK(eo_shape(G, {&out, &w, &x}, "schur_dot"));
  if (x.prec != out.prec) return fail(MGLMA_ERR_INVALID, "schur_dot: fields of one precision needed");
  if (out.nrhs == 0) return MGLMA_OK;
  EvArgs a;
  a.part = part;
  {
    const bool bf = out.prec == MGLMA_BF16;
    ProfScope ps(ctx, K_DSLASH32, s, schur_bytes(G, out.nrhs, bf ? 192.0 : 288.0), schur_flops(G, out.nrhs));
    if (bf)
      launch_even<EV_DOT>(G, w, x.p, out.p, a, s);
    else
      launch_even<EV_DOT, float>(G, w, x.p, out.p, a, s);
  }
  MG_LAUNCH_CHECK();
  return mr_finish(ctx, G, part, out.nrhs, alpha, s);
}

mglma_status schur_mr_step(mglma_ctx ctx, const mglma_gauge_s* G, const Spinor& w, const Spinor& t, Spinor& tn,
                           const Spinor& sk, Spinor& sn, const float2* alpha, float2* alpha_n, double* part,
                           cudaStream_t s) {
  MG_CHECK(eo_shape(G, {&tn, &w, &t, &sk, &sn}, "schur_mr_step"));
  if (t.prec != tn.prec || sk.prec != tn.prec || sn.prec != tn.prec)
    return fail(MGLMA_ERR_INVALID, "schur_mr_step: fields of one precision needed");
  if (tn.nrhs == 0) return MGLMA_OK;
  EvArgs a;
  a.s = sk.p;
  a.sn = sn.p;
  a.alpha = alpha;
  a.part = part;
  {
    const bool bf = tn.prec == MGLMA_BF16;
    ProfScope ps(ctx, K_DSLASH32, s, schur_bytes(G, tn.nrhs, bf ? 288.0 : 480.0), schur_flops(G, tn.nrhs));
    if (bf)
      launch_even<EV_MR>(G, w, t.p, tn.p, a, s);
    else
      launch_even<EV_MR, float>(G, w, t.p, tn.p, a, s);
  }
  MG_LAUNCH_CHECK();
  return mr_finish(ctx, G, part, tn.nrhs, alpha_n, s);
}

template <typename SM>
static mglma_status launch_iterate(Spinor& z, const uint4* sp, size_t st, int ns, const float2* alpha,
                                   cudaStream_t s) {
  const uint32_t Vh = (uint32_t)z.V;
  const dim3 g((Vh + 255) / 256, z.nrhs, 3);
  switch (ns) {
    case 1: mr_iterate_kernel<1, SM><<<g, 256, 0, s>>>((float4*)z.p, sp, st, alpha, z.nrhs, Vh); break;
    case 2: mr_iterate_kernel<2, SM><<<g, 256, 0, s>>>((float4*)z.p, sp, st, alpha, z.nrhs, Vh); break;
    case 3: mr_iterate_kernel<3, SM><<<g, 256, 0, s>>>((float4*)z.p, sp, st, alpha, z.nrhs, Vh); break;
    case 4: mr_iterate_kernel<4, SM><<<g, 256, 0, s>>>((float4*)z.p, sp, st, alpha, z.nrhs, Vh); break;
    default: return fail(MGLMA_ERR_INVALID, "mr_iterate: 1 to 4 steps");
  }
  MG_LAUNCH_CHECK();
  return MGLMA_OK;
}

mglma_status mr_iterate(mglma_ctx ctx, Spinor& z, const void* s0, int sprec, size_t sstride_bytes, int ns,
                        const float2* alpha, cudaStream_t s) {
  if (z.nrhs == 0) return MGLMA_OK;
  const bool bf = sprec == MGLMA_BF16;
  ProfScope ps(ctx, K_BLAS, s, (192.0 + (bf ? 48.0 : 96.0) * ns) * (double)z.V * z.nrhs);
  if (bf) return launch_iterate<SpinBf16>(z, (const uint4*)s0, sstride_bytes / 16, ns, alpha, s);
  return launch_iterate<float>(z, (const uint4*)s0, sstride_bytes / 16, ns, alpha, s);
}

mglma_status schur_gcr(mglma_ctx ctx, const mglma_gauge_s* G, const Spinor& w, const Spinor& x, Spinor& out, int k,
                       const void* W0, size_t wslot_reals, const void* r, double* part, double* nw, double2* num,
                       double2* dots, cudaStream_t s) {
  MG_CHECK(eo_shape(G, {&out, &w, &x}, "schur_gcr"));
  if (k < 0 || k > 3) return fail(MGLMA_ERR_INVALID, "schur_gcr: 0 to 3 earlier directions");
  if (out.nrhs == 0) return MGLMA_OK;
  EvArgs a;
  a.part = part;
  a.W0 = (const char*)W0;
  a.wslot = wslot_reals * sizeof(float);
  a.k = k;
  a.r = r;
  {
    ProfScope ps(ctx, K_DSLASH32, s, schur_bytes(G, out.nrhs, 288.0 + 96.0 * (k ? k : 1)), schur_flops(G, out.nrhs));
    launch_even<EV_GCR>(G, w, x.p, out.p, a, s);
  }
  MG_LAUNCH_CHECK();
  return gd_finish(ctx, part, schur_blocks(G), k, out.nrhs, nw, num, dots, s);
}

static dim3 half_grid(const mglma_gauge_s* G, int nrhs) {
  return dim3((unsigned)((G->g.V / 2 + 127) / 128), (unsigned)nrhs, 1);
}

mglma_status eo_split(mglma_ctx ctx, const mglma_gauge_s* G, const Spinor& f, Spinor& e, Spinor& o,
                      const double* scale, cudaStream_t s) {
  MG_CHECK(eo_shape(G, {&e, &o}, "eo_split"));
  ProfScope ps(ctx, K_PACK, s, 288.0 * (double)f.V * f.nrhs);
  eo_split_kernel<<<half_grid(G, f.nrhs), 128, 0, s>>>((const double2*)f.p, (float4*)e.p, (float4*)o.p,
                                                       make_eogeo(G->g.L), scale);
  MG_LAUNCH_CHECK();
  return MGLMA_OK;
}

mglma_status eo_join(mglma_ctx ctx, const mglma_gauge_s* G, const Spinor& e, const Spinor& o, Spinor& f, Spinor& x,
                     const double* scale, cudaStream_t s) {
  MG_CHECK(eo_shape(G, {&e, &o}, "eo_join"));
  ProfScope ps(ctx, K_PACK, s, 576.0 * (double)f.V * f.nrhs);
  eo_join_kernel<<<half_grid(G, f.nrhs), 128, 0, s>>>((const float4*)e.p, (const float4*)o.p, (float4*)f.p,
                                                      (double2*)x.p, make_eogeo(G->g.L), scale);
  MG_LAUNCH_CHECK();
  return MGLMA_OK;
}

mglma_status eo_embed(mglma_ctx ctx, const mglma_gauge_s* G, const Spinor& e, Spinor& f, cudaStream_t s) {
  MG_CHECK(eo_shape(G, {&e}, "eo_embed"));
  ProfScope ps(ctx, K_PACK, s, 144.0 * (double)f.V * f.nrhs);
  eo_embed_kernel<<<half_grid(G, f.nrhs), 128, 0, s>>>((const float4*)e.p, (float4*)f.p, make_eogeo(G->g.L));
  MG_LAUNCH_CHECK();
  return MGLMA_OK;
}

mglma_status eo_extract(mglma_ctx ctx, const mglma_gauge_s* G, const Spinor& f, Spinor& e, cudaStream_t s) {
  MG_CHECK(eo_shape(G, {&e}, "eo_extract"));
  ProfScope ps(ctx, K_PACK, s, 144.0 * (double)f.V * f.nrhs);
  eo_extract_kernel<<<half_grid(G, f.nrhs), 128, 0, s>>>((const float4*)f.p, (float4*)e.p, make_eogeo(G->g.L));
  MG_LAUNCH_CHECK();
  return MGLMA_OK;
}

}  // namespace mglma
