// Inverse of a packed Hermitian 6x6 clover block in registers (one thread).
#pragma once
#include "stencil.cuh"

namespace mglma {

// elimination step K: pivot search in column K, exchange, scaling, reduction.  The
// step is a template so that every index of M is a constant
template <int K>
__device__ __forceinline__ void clover_eliminate(Cx<double> (&M)[6][6], int (&perm)[6], bool& ok) {
  int p = K;
  double best = M[K][K].re * M[K][K].re + M[K][K].im * M[K][K].im;
#pragma unroll
  for (int r = K + 1; r < 6; ++r) {
    const double m = M[r][K].re * M[r][K].re + M[r][K].im * M[r][K].im;
    if (m > best) {
      best = m;
      p = r;
    }
  }
  perm[K] = p;
  ok = ok && best > 0;
#pragma unroll
  for (int r = K + 1; r < 6; ++r) {
    const bool e = r == p;
#pragma unroll
    for (int j = 0; j < 6; ++j) {
      const Cx<double> a = M[K][j], b = M[r][j];
      M[K][j] = cx(e ? b.re : a.re, e ? b.im : a.im);
      M[r][j] = cx(e ? a.re : b.re, e ? a.im : b.im);
    }
  }
  const double m = M[K][K].re * M[K][K].re + M[K][K].im * M[K][K].im;
  // singular: finish with harmless numbers, reported by ok
  const Cx<double> d = m > 0 ? cx(M[K][K].re / m, -M[K][K].im / m) : cx(0.0, 0.0);
#pragma unroll
  for (int j = 0; j < 6; ++j)
    if (j != K) M[K][j] = M[K][j] * d;
#pragma unroll
  for (int r = 0; r < 6; ++r)
    if (r != K) {
      const Cx<double> f = M[r][K];
#pragma unroll
      for (int j = 0; j < 6; ++j)
        if (j != K) M[r][j] = M[r][j] - f * M[K][j];
      M[r][K] = -(f * d);
    }
  M[K][K] = d;
}

// the exchange of step K undone, as a column exchange (last step first)
template <int K>
__device__ __forceinline__ void clover_unexchange(Cx<double> (&M)[6][6], const int (&perm)[6]) {
#pragma unroll
  for (int c = K + 1; c < 6; ++c) {
    const bool e = perm[K] == c;
#pragma unroll
    for (int r = 0; r < 6; ++r) {
      const Cx<double> a = M[r][K], b = M[r][c];
      M[r][K] = cx(e ? b.re : a.re, e ? b.im : a.im);
      M[r][c] = cx(e ? a.re : b.re, e ? a.im : b.im);
    }
  }
}

// pk = c^-1 by Gauss-Jordan with partial pivoting in FP64; the inverse of a
// Hermitian matrix is Hermitian and is packed the same way.  Row and column
// exchanges are selections and every index is a constant, so the 6x6 matrix stays
// in registers (254, no stack; as one loop over the steps the compiler kept it in
// 576 bytes of local memory).  An earlier version that indexed the array by the
// pivot row gave wrong inverses under -O3 for a cause never found.  False when the
// block is singular.
__device__ __forceinline__ bool clover_inverse6(const double c[36], double pk[36]) {
  Cx<double> M[6][6];
#pragma unroll
  for (int i = 0; i < 6; ++i) {
    M[i][i] = cx(c[i], 0.0);
#pragma unroll
    for (int j = 0; j < 6; ++j) {
      if (j <= i) continue;
      const int k = 6 + 2 * offdiag_slot(i, j);
      M[i][j] = cx(c[k], c[k + 1]);
      M[j][i] = cx(c[k], -c[k + 1]);
    }
  }
  int perm[6];
  bool ok = true;
  clover_eliminate<0>(M, perm, ok);
  clover_eliminate<1>(M, perm, ok);
  clover_eliminate<2>(M, perm, ok);
  clover_eliminate<3>(M, perm, ok);
  clover_eliminate<4>(M, perm, ok);
  clover_eliminate<5>(M, perm, ok);
  clover_unexchange<4>(M, perm);
  clover_unexchange<3>(M, perm);
  clover_unexchange<2>(M, perm);
  clover_unexchange<1>(M, perm);
  clover_unexchange<0>(M, perm);
#pragma unroll
  for (int i = 0; i < 6; ++i) {
    pk[i] = M[i][i].re;
#pragma unroll
    for (int j = 0; j < 6; ++j) {
      if (j <= i) continue;
      const int k = 6 + 2 * offdiag_slot(i, j);
      pk[k] = M[i][j].re;
      pk[k + 1] = M[i][j].im;
    }
  }
  return ok;
}

}  // namespace mglma
