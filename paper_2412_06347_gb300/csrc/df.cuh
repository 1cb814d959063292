// Double-float ("double-word") arithmetic: a real as an unevaluated sum
// hi + lo of two FP32 numbers with |lo| <= ulp(hi) / 2, about 48 significant
// bits.  GB300 runs FP32 at many times its FP64 rate, so a stencil that must
// reach FP64-level accuracy on FP32 inputs runs faster in this form.
//
// Building blocks (exact error-free transformations of IEEE binary32):
//   two_sum(a, b)      = (s, e), s = fl(a + b), a + b = s + e exactly
//                        (Knuth's branch-free form, six operations)
//   fast_two_sum(a, b) = the same for |a| >= |b| (Dekker, three operations)
//   two_prod(a, b)     = (p, e), p = fl(a b), a b = p + e exactly, e taken
//                        by one fused multiply-add
// Sums use the "sloppy" double-word addition (exact sum of the high parts,
// low parts added in FP32, renormalised): its error is a small multiple of
// 2^-48 (|x| + |y|), i.e. bounded by the operands, not by the result -- the
// same kind of bound an FP64 sum has, which is what a stencil sum needs.
// Products keep the cross terms hi lo by FMA and drop lo lo (below 2^-48).
//
// The type and its operators live in a namespace of their own so that only
// argument-dependent lookup finds them: an unqualified fma on FP32 or FP64
// arguments keeps resolving to CUDA's own.
#pragma once
#include <cuda_runtime.h>

#include <cmath>

namespace mglma {
namespace dfl {

struct DF {
  float hi, lo;
  __host__ __device__ DF() : hi(0.f), lo(0.f) {}
  __host__ __device__ DF(float h, float l) : hi(h), lo(l) {}
  // d split into FP32 high and low parts (within 2^-48 relative of d for d
  // inside the FP32 exponent range)
  __host__ __device__ DF(double d) : hi((float)d), lo((float)(d - (double)(float)d)) {}
  __host__ __device__ DF(int i) : DF((double)i) {}
};

// FP32 operations the compiler may neither contract into an FMA nor
// reorder (device: the _rn intrinsics; host: plain operators, built without
// contraction), on one value or on a packed pair of them, lane by lane.  A pair
// has no subtraction of its own: b (-1) is exact, so a + b (-1) rounds like a - b.
__host__ __device__ __forceinline__ float df_add(float a, float b) {
#ifdef __CUDA_ARCH__
  return __fadd_rn(a, b);
#else
  return a + b;
#endif
}
__host__ __device__ __forceinline__ float df_sub(float a, float b) {
#ifdef __CUDA_ARCH__
  return __fsub_rn(a, b);
#else
  return a - b;
#endif
}
__host__ __device__ __forceinline__ float df_mul(float a, float b) {
#ifdef __CUDA_ARCH__
  return __fmul_rn(a, b);
#else
  return a * b;
#endif
}
__host__ __device__ __forceinline__ float df_fma(float a, float b, float c) { return fmaf(a, b, c); }
__host__ __device__ __forceinline__ float df_neg(float a) { return -a; }
__host__ __device__ __forceinline__ float2 df_add(float2 a, float2 b) {
#ifdef __CUDA_ARCH__
  return __fadd2_rn(a, b);
#else
  return make_float2(a.x + b.x, a.y + b.y);
#endif
}
__host__ __device__ __forceinline__ float2 df_mul(float2 a, float2 b) {
#ifdef __CUDA_ARCH__
  return __fmul2_rn(a, b);
#else
  return make_float2(a.x * b.x, a.y * b.y);
#endif
}
__host__ __device__ __forceinline__ float2 df_fma(float2 a, float2 b, float2 c) {
#ifdef __CUDA_ARCH__
  return __ffma2_rn(a, b, c);
#else
  return make_float2(fmaf(a.x, b.x, c.x), fmaf(a.y, b.y, c.y));
#endif
}
__host__ __device__ __forceinline__ float2 df_sub(float2 a, float2 b) { return df_fma(b, make_float2(-1.f, -1.f), a); }
__host__ __device__ __forceinline__ float2 df_neg(float2 a) { return make_float2(-a.x, -a.y); }

// The arithmetic, once for both: F is float (D = DF) or float2 (D = DF2).
template <typename D, typename F>
__host__ __device__ __forceinline__ D two_sum_of(F a, F b) {
  const F s = df_add(a, b), bb = df_sub(s, a);
  return D(s, df_add(df_sub(a, df_sub(s, bb)), df_sub(b, bb)));
}
template <typename D, typename F>
__host__ __device__ __forceinline__ D fast_two_sum_of(F a, F b) {
  const F s = df_add(a, b);
  return D(s, df_sub(b, df_sub(s, a)));
}
template <typename D>
__host__ __device__ __forceinline__ D add_of(D x, D y) {
  const D s = two_sum_of<D>(x.hi, y.hi);
  return fast_two_sum_of<D>(s.hi, df_add(s.lo, df_add(x.lo, y.lo)));
}
// x y + z with one renormalisation; t is minus the product's rounding error and
// its cross terms (the negated x serves several products where it is loop-invariant)
template <typename D>
__host__ __device__ __forceinline__ D fma_of(D x, D y, D z) {
  const auto nh = df_neg(x.hi), nl = df_neg(x.lo);
  const auto p = df_mul(x.hi, y.hi);
  const auto t = df_fma(nh, y.lo, df_fma(nl, y.hi, df_fma(nh, y.hi, p)));
  const D s = two_sum_of<D>(p, z.hi);
  return fast_two_sum_of<D>(s.hi, df_add(s.lo, df_sub(z.lo, t)));
}
// the same for FP32 y
template <typename D, typename F>
__host__ __device__ __forceinline__ D fma_single_of(D x, F y, D z) {
  const auto nh = df_neg(x.hi), nl = df_neg(x.lo);
  const auto p = df_mul(x.hi, y);
  const auto t = df_fma(nl, y, df_fma(nh, y, p));
  const D s = two_sum_of<D>(p, z.hi);
  return fast_two_sum_of<D>(s.hi, df_add(s.lo, df_sub(z.lo, t)));
}

__host__ __device__ __forceinline__ DF two_sum(float a, float b) { return two_sum_of<DF>(a, b); }
__host__ __device__ __forceinline__ DF fast_two_sum(float a, float b) { return fast_two_sum_of<DF>(a, b); }
__host__ __device__ __forceinline__ DF two_prod(float a, float b) {
  const float p = df_mul(a, b);
  return DF(p, fmaf(a, b, -p));
}
__host__ __device__ __forceinline__ DF operator+(DF x, DF y) { return add_of(x, y); }
__host__ __device__ __forceinline__ DF operator-(DF x) { return DF(-x.hi, -x.lo); }
__host__ __device__ __forceinline__ DF operator-(DF x, DF y) { return x + (-y); }
__host__ __device__ __forceinline__ DF operator*(DF x, DF y) {
  const DF p = two_prod(x.hi, y.hi);
  return fast_two_sum(p.hi, fmaf(x.hi, y.lo, fmaf(x.lo, y.hi, p.lo)));
}
__host__ __device__ __forceinline__ DF fma(DF x, DF y, DF z) { return fma_of(x, y, z); }
__host__ __device__ __forceinline__ DF fma(DF x, float y, DF z) { return fma_single_of(x, y, z); }

// two double-floats in the lanes of packed pairs (resid_df.cu)
struct DF2 {
  float2 hi, lo;
  __host__ __device__ DF2() : hi(make_float2(0.f, 0.f)), lo(make_float2(0.f, 0.f)) {}
  __host__ __device__ DF2(float2 h, float2 l) : hi(h), lo(l) {}
};
__host__ __device__ __forceinline__ DF2 two_sum(float2 a, float2 b) { return two_sum_of<DF2>(a, b); }
__host__ __device__ __forceinline__ DF2 operator+(DF2 x, DF2 y) { return add_of(x, y); }
__host__ __device__ __forceinline__ DF2 fma(DF2 x, DF2 y, DF2 z) { return fma_of(x, y, z); }
__host__ __device__ __forceinline__ DF2 fma(DF2 x, float2 y, DF2 z) { return fma_single_of(x, y, z); }

// hi + lo rounded once to FP64
__host__ __device__ __forceinline__ double to_double(DF x) { return (double)x.hi + (double)x.lo; }

}  // namespace dfl
using dfl::DF;
using dfl::DF2;
}  // namespace mglma
