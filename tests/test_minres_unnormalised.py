"""The MINRES scalar recurrence on unnormalised Lanczos vectors (csrc/minres.cuh),
built for the host and driven with the vector steps of the coarse kernel,
including its pending update (iteration k's direction and iterate are formed
during iteration k + 1): on a complex Hermitian indefinite matrix |eta| is the
true residual at every iteration and n iterations reach numpy's solution."""
import os
import shutil
import subprocess

import numpy as np
import pytest

from test_minres_recurrence import CSRC, CUDA_INC, _hermitian_indefinite, _run

PROG = r"""
#include <complex>
#include <cstdio>
#include <vector>
#include "minres.cuh"
using namespace mglma;
typedef std::complex<double> C;
int main() {
  int n, iters;
  if (std::scanf("%d %d", &n, &iters) != 2) return 1;
  std::vector<C> A(n * n), b(n);
  for (auto& a : A) { double re, im; std::scanf("%lf %lf", &re, &im); a = C(re, im); }
  for (auto& v : b) { double re, im; std::scanf("%lf %lf", &re, &im); v = C(re, im); }
  std::vector<double> st(MR_COUNT, 0.0);
  auto S = [&](int j) -> double& { return st[j]; };
  int active = 1;
  double bb = 0;
  for (auto& v : b) bb += std::norm(v);
  const double b1 = std::sqrt(bb);
  S(MR_BETA1) = S(MR_ETA) = b1; S(MR_C2) = S(MR_C1) = 1; S(MR_LC) = 1; S(MR_LC + 1) = -1;
  std::vector<C> u(n), uo(n, 0.0), y(n), w[2] = {std::vector<C>(n, 0.0), std::vector<C>(n, 0.0)}, x(n, 0.0);
  for (int i = 0; i < n; ++i) u[i] = b[i] / b1;
  auto pending = [&](const std::vector<C>& v, int k) {  // iteration k's update, v = u_k
    for (int i = 0; i < n; ++i) {
      w[k % 2][i] = S(MR_CF) * v[i] + S(MR_CF + 1) * w[(k + 1) % 2][i] + S(MR_CF + 2) * w[k % 2][i];
      x[i] += S(MR_CF + 3) * w[k % 2][i];
    }
  };
  double eta = b1;
  for (int k = 0; k <= iters; ++k) {
    if (k > 0 && S(MR_CF + 5) != 0.0) {
      pending(uo, k - 1);
      std::printf("eta %d %.17g\n", k - 1, std::fabs(eta));
      for (int i = 0; i < n; ++i) std::printf("x %d %d %.17g %.17g\n", k - 1, i, x[i].real(), x[i].imag());
    }
    if (!active || k == iters) break;
    for (int i = 0; i < n; ++i) { y[i] = 0; for (int j = 0; j < n; ++j) y[i] += A[i * n + j] * u[j]; }
    double dot = 0, zz = 0;
    for (int i = 0; i < n; ++i) dot += (std::conj(u[i]) * y[i]).real();
    for (int i = 0; i < n; ++i) {
      y[i] = S(MR_LC) * y[i] + dot * S(MR_LC + 1) * u[i] + S(MR_LC + 2) * uo[i];
      zz += std::norm(y[i]);
    }
    S(MR_BN2) = zz;
    minres_scalar_step_u(st.data(), dot, &active, 0.0, 1, 0);
    eta = S(MR_ETA);
    uo = u;
    u = y;
  }
  return 0;
}
"""


@pytest.fixture(scope="module")
def exe(tmp_path_factory):
    gxx = shutil.which("g++")
    if not gxx or not os.path.isfile(os.path.join(CUDA_INC, "cuda_runtime.h")):
        pytest.skip("g++ or the CUDA headers are missing")
    d = tmp_path_factory.mktemp("minres_u")
    src, out = d / "t.cpp", d / "t"
    src.write_text(PROG)
    subprocess.run([gxx, "-std=c++17", "-O2", "-I", CSRC, "-I", CUDA_INC, str(src), "-o", str(out)], check=True,
                   capture_output=True)
    return str(out)


@pytest.mark.parametrize("n,seed", [(24, 5), (16, 9), (1, 3)])
def test_residual_and_solution(exe, n, seed):
    A, b = _hermitian_indefinite(n, seed)
    eta, xs = _run(exe, A, b, n)
    nb = np.linalg.norm(b)
    for k in sorted(eta):
        assert abs(eta[k] - np.linalg.norm(b - A @ xs[k])) <= 1e-10 * nb
    want = np.linalg.solve(A, b)
    assert np.linalg.norm(xs[max(xs)] - want) <= 1e-9 * np.linalg.norm(want)
