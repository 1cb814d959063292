"""The packed double-float operations of the residual update (csrc/df.cuh, DF2), on
the host: lane by lane the same bits as the scalar ones, the FP32-operand product
within the same bound, and the lanes independent of each other."""
import os
import shutil
import subprocess
from fractions import Fraction

import pytest

from test_df_arith import CSRC, CUDA_INC, _pairs

PROG = r"""
#include <cstdio>
#include <cstdint>
#include <cmath>
#include "df.cuh"
using mglma::DF;
using mglma::DF2;
namespace d = mglma::dfl;
static uint64_t st = 0x2545F4914F6CDD1Dull;
static double val() {
  auto u = [] {
    st = st * 6364136223846793005ull + 1442695040888963407ull;
    return (double)(st >> 11) * (1.0 / 9007199254740992.0);
  };
  const double m = 2.0 * u() - 1.0;
  return m * std::pow(10.0, 6.0 * u() - 3.0);
}
static DF2 pack(DF a, DF b) { return DF2(make_float2(a.hi, b.hi), make_float2(a.lo, b.lo)); }
static bool same(DF2 p, DF a, DF b) { return p.hi.x == a.hi && p.hi.y == b.hi && p.lo.x == a.lo && p.lo.y == b.lo; }
static void pr(const char* tag, DF x) { std::printf(" %s %a %a", tag, (double)x.hi, (double)x.lo); }
int main() {
  for (int i = 0; i < 4000; ++i) {
    DF x[2], y[2], z[2];
    for (int l = 0; l < 2; ++l) {
      x[l] = DF(val()); y[l] = DF(val()); z[l] = DF(val());
      if (i % 4 == 1) y[l] = -x[l] + DF(val() * 1e-9);       // near-cancelling sums
      if (i % 4 == 2) z[l] = -(x[l] * y[l]) + DF(val() * 1e-7);
    }
    const DF2 X = pack(x[0], x[1]), Y = pack(y[0], y[1]), Z = pack(z[0], z[1]);
    const bool ok = same(d::two_sum(X.hi, Y.hi), d::two_sum(x[0].hi, y[0].hi), d::two_sum(x[1].hi, y[1].hi)) &&
                    same(X + Y, x[0] + y[0], x[1] + y[1]) &&
                    same(fma(X, Y, Z), fma(x[0], y[0], z[0]), fma(x[1], y[1], z[1])) &&
                    same(fma(X, Y.hi, Z), fma(x[0], y[0].hi, z[0]), fma(x[1], y[1].hi, z[1]));
    for (int l = 0; l < 2; ++l) {
      std::printf("%d", ok ? 1 : 0);
      pr("x", x[l]); pr("y", DF(y[l].hi, 0.f)); pr("z", z[l]);
      pr("fs", fma(x[l], y[l].hi, z[l]));
      std::printf("\n");
    }
  }
  return 0;
}
"""


def test_pairs(tmp_path):
    gxx = shutil.which("g++")
    if not gxx or not os.path.isfile(os.path.join(CUDA_INC, "cuda_runtime.h")):
        pytest.skip("g++ or the CUDA headers are missing")
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(PROG)
    subprocess.run([gxx, "-std=c++17", "-O2", "-ffp-contract=off", "-I", CSRC, "-I", CUDA_INC, str(src), "-o",
                    str(exe)], check=True, capture_output=True)
    lines = [ln.split() for ln in subprocess.run([str(exe)], check=True, capture_output=True,
                                                 text=True).stdout.splitlines()]
    assert len(lines) == 8000
    eps = Fraction(1, 2**45)
    for t in lines:
        assert t[0] == "1"
        x, y, z = (sum(_pairs(t, k)) for k in ("x", "y", "z"))
        assert abs(sum(_pairs(t, "fs")) - (x * y + z)) <= eps * (abs(x * y) + abs(z))
