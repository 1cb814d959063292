// Inverse of a packed Hermitian 6x6 clover block (one thread).
#pragma once
#include "stencil.cuh"

namespace mglma {

// pk = c^-1 by Gauss-Jordan with partial pivoting in FP64; the inverse of a
// Hermitian matrix is Hermitian and is packed the same way.  Every loop is
// unrolled and every index static (row and column exchanges are predicated
// swaps); ptxas keeps 576 bytes of it in local memory all the same (254 registers),
// which a set-up kernel can afford.  An earlier version that indexed the array by
// the pivot row gave wrong inverses under -O3 for a cause never found;
// tests/test_gpu_clover_inverse.py holds blocks whose rows are exchanged.  False
// when the block is singular.
__device__ __forceinline__ bool clover_inverse6(const double c[36], double pk[36]) {
  Cx<double> M[6][6];
#pragma unroll
  for (int i = 0; i < 6; ++i) M[i][i] = cx(c[i], 0.0);
#pragma unroll
  for (int i = 0; i < 6; ++i)
#pragma unroll
    for (int j = i + 1; j < 6; ++j) {
      const int k = 6 + 2 * offdiag_slot(i, j);
      M[i][j] = cx(c[k], c[k + 1]);
      M[j][i] = cx(c[k], -c[k + 1]);
    }
  int perm[6];
  bool ok = true;
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    int p = k;
    double best = M[k][k].re * M[k][k].re + M[k][k].im * M[k][k].im;
#pragma unroll
    for (int r = k + 1; r < 6; ++r) {
      const double m = M[r][k].re * M[r][k].re + M[r][k].im * M[r][k].im;
      if (m > best) {
        best = m;
        p = r;
      }
    }
    perm[k] = p;
    ok = ok && best > 0;
    if (!(best > 0)) best = 1;  // singular: finish with harmless numbers, report below
#pragma unroll
    for (int r = k + 1; r < 6; ++r)
      if (r == p)
#pragma unroll
        for (int j = 0; j < 6; ++j) {
          const Cx<double> tmp = M[k][j];
          M[k][j] = M[r][j];
          M[r][j] = tmp;
        }
    const double m = M[k][k].re * M[k][k].re + M[k][k].im * M[k][k].im;
    const Cx<double> d = m > 0 ? cx(M[k][k].re / m, -M[k][k].im / m) : cx(0.0, 0.0);
#pragma unroll
    for (int j = 0; j < 6; ++j)
      if (j != k) M[k][j] = M[k][j] * d;
#pragma unroll
    for (int r = 0; r < 6; ++r) {
      if (r == k) continue;
      const Cx<double> f = M[r][k];
#pragma unroll
      for (int j = 0; j < 6; ++j)
        if (j != k) M[r][j] = M[r][j] - f * M[k][j];
      M[r][k] = -(f * d);
    }
    M[k][k] = d;
  }
  // undo the row exchanges as column exchanges, last first
#pragma unroll
  for (int k = 5; k >= 0; --k)
#pragma unroll
    for (int c2 = k + 1; c2 < 6; ++c2)
      if (perm[k] == c2)
#pragma unroll
        for (int r = 0; r < 6; ++r) {
          const Cx<double> tmp = M[r][k];
          M[r][k] = M[r][c2];
          M[r][c2] = tmp;
        }
#pragma unroll
  for (int i = 0; i < 6; ++i) pk[i] = M[i][i].re;
#pragma unroll
  for (int i = 0; i < 6; ++i)
#pragma unroll
    for (int j = i + 1; j < 6; ++j) {
      const int k = 6 + 2 * offdiag_slot(i, j);
      pk[k] = M[i][j].re;
      pk[k + 1] = M[i][j].im;
    }
  return ok;
}

}  // namespace mglma
