// Per-RHS scalar recurrence of the batched coarse MINRES (Givens QR of the
// Lanczos tridiagonal), shared by its own kernel and by the Lanczos-norm
// kernel that runs it in its last block.  State layout: st[j * cap + r] for
// the slots below.
#pragma once
#include <cuda_runtime.h>

#include <cmath>

namespace mglma {

enum {
  MR_BETA1 = 0,
  MR_ETA,
  MR_BETA,
  MR_C2,
  MR_S2,
  MR_C1,
  MR_S1,
  MR_BN2,
  MR_BB,
  MR_CF,  // six update coefficients (minres_update), MR_CF + 4 also scales v_0
  MR_LC = MR_CF + 6,  // unnormalised form: 1 / b_k, -1 / b_k^3, -beta_k / b_(k-1)
  MR_COUNT = MR_LC + 3
};

// alpha = Re dot[r] = <v_k, Qhat v_k>, |z|^2 in slot MR_BN2: the rotation of
// iteration k, the update coefficients (MR_CF .. MR_CF + 5; MR_CF + 5 = 1
// when the update applies) and the new activity of RHS r
__host__ __device__ __forceinline__ void minres_scalar_step(double* st, const double2* dot, int* active, double tol,
                                                            int cap, int r) {
  auto S = [&](int j) -> double& { return st[(size_t)j * cap + r]; };
  S(MR_CF + 5) = 0;
  if (!active[r]) return;
  const double alpha = dot[r].x, beta = S(MR_BETA);
  const double bn = sqrt(fmax(S(MR_BN2), 0.0));
  const double eps = S(MR_S2) * beta, dp = S(MR_C2) * beta;
  const double delta = S(MR_C1) * dp + S(MR_S1) * alpha;
  const double gp = S(MR_C1) * alpha - S(MR_S1) * dp;
  const double gamma = hypot(gp, bn);
  if (!(gamma > 0) || !(gamma < INFINITY)) {  // breakdown: keep the iterate
    active[r] = 0;
    return;
  }
  const double c = gp / gamma, sn = bn / gamma;
  S(MR_CF + 0) = 1.0 / gamma;
  S(MR_CF + 1) = -delta / gamma;
  S(MR_CF + 2) = -eps / gamma;
  S(MR_CF + 3) = c * S(MR_ETA);
  S(MR_CF + 4) = bn > 0 ? 1.0 / bn : 0.0;
  S(MR_CF + 5) = 1;
  S(MR_ETA) = -sn * S(MR_ETA);
  S(MR_C2) = S(MR_C1);
  S(MR_S2) = S(MR_S1);
  S(MR_C1) = c;
  S(MR_S1) = sn;
  S(MR_BETA) = bn;
  active[r] = (bn > 0 && fabs(S(MR_ETA)) > tol * S(MR_BETA1)) ? 1 : 0;
}

// The same recurrence on unnormalised Lanczos vectors u_k = b_k v_k (u_0 = v_0, b_0
// = 1), so that a vector can enter the operator before its norm is known:
//   u_(k+1) = c1 Q u_k + c2 u_k + c3 u_(k-1),  c1 = st[MR_LC], c2 = dot st[MR_LC + 1],
//   c3 = st[MR_LC + 2], dot = Re <u_k, Q u_k>, and b_(k+1)^2 = |u_(k+1)|^2 in MR_BN2
// Afterwards MR_CF .. MR_CF + 3 are the coefficients of iteration k's update
//   w_k = cf0 u_k + cf1 w_(k-1) + cf2 w_(k-2),  x += cf3 w_k  (when cf5 = 1)
// and MR_LC .. those of the next iteration.  The reciprocal square roots replace
// a hypot, two square roots and six divisions: one thread runs this between two
// launches, on an FP64 pipe where each of those is a long dependent chain.
__host__ __device__ __forceinline__ double minres_rsqrt(double a) {
#ifdef __CUDA_ARCH__
  return rsqrt(a);
#else
  return 1.0 / sqrt(a);
#endif
}
__host__ __device__ __forceinline__ void minres_scalar_step_u(double* st, double dot, int* active, double tol, int cap,
                                                              int r) {
  auto S = [&](int j) -> double& { return st[(size_t)j * cap + r]; };
  S(MR_CF + 5) = 0;
  if (!active[r]) return;
  const double ib = S(MR_LC), beta = S(MR_BETA), alpha = dot * ib * ib;
  const double bn2 = fmax(S(MR_BN2), 0.0), ibn = bn2 > 0 ? minres_rsqrt(bn2) : 0.0, bn = bn2 * ibn;
  const double eps = S(MR_S2) * beta, dp = S(MR_C2) * beta;
  const double delta = S(MR_C1) * dp + S(MR_S1) * alpha;
  const double gp = S(MR_C1) * alpha - S(MR_S1) * dp;
  const double g2 = gp * gp + bn2;
  if (!(g2 > 0) || !(g2 < INFINITY)) {  // breakdown: keep the iterate
    active[r] = 0;
    return;
  }
  const double ig = minres_rsqrt(g2), c = gp * ig, sn = bn * ig;
  S(MR_CF + 0) = ig * ib;
  S(MR_CF + 1) = -delta * ig;
  S(MR_CF + 2) = -eps * ig;
  S(MR_CF + 3) = c * S(MR_ETA);
  S(MR_CF + 5) = 1;
  S(MR_ETA) = -sn * S(MR_ETA);
  S(MR_C2) = S(MR_C1);
  S(MR_S2) = S(MR_S1);
  S(MR_C1) = c;
  S(MR_S1) = sn;
  S(MR_BETA) = bn;
  S(MR_LC) = ibn;
  S(MR_LC + 1) = -ibn * ibn * ibn;
  S(MR_LC + 2) = -bn * ib;
  active[r] = (bn > 0 && fabs(S(MR_ETA)) > tol * S(MR_BETA1)) ? 1 : 0;
}

}  // namespace mglma
