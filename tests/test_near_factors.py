"""The FP64 near sums' factor polynomials (csrc/sk_near_factors.h): s1/rho,
s2/rho^3 and s3/rho^5 for rho^2 < 1/4, evaluated as the kernels evaluate them
(compiled with the host compiler) against 40-digit closed forms. Bound 2e-15: the
coefficients come from at most 18 rounded series terms and the evaluation rounds
five times in FP64 (2^-53 each); the FP32 terms from t^5 on are below 2^-36 of the
factor and round at 2^-24.
"""

import os
import shutil
import subprocess

import numpy as np
import pytest

from test_factors64 import exact_factor

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2310_13908_gb300", "csrc")

PROGRAM = r"""
#include <cmath>
#include <cstdio>
#include "sk_near_factors.h"
using namespace sk;
int main() {
  static constexpr NearFactors f = near_factors();
  double x;
  while (std::scanf("%lf", &x) == 1)
    for (int w = 0; w < 3; ++w) {
      const double H = NEAR_X_MAX / NEAR_N;
      int i = (int)((float)x * (float)(1.0 / H));
      if (i > NEAR_N - 1) i = NEAR_N - 1;
      const double t = x - (double)(((float)i + 0.5f) * (float)H);
      const float tf = (float)t;
      const float v = std::fma(std::fma(f.t[w][2][i], tf, f.t[w][1][i]), tf, f.t[w][0][i]) * tf;
      double p = f.c[w][4][i] + (double)v;
      for (int k = 3; k >= 0; --k) p = std::fma(p, t, f.c[w][k][i]);
      std::printf("%.17g\n", p);
    }
}
"""


def test_near_factors_match_closed_forms(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("needs a host C++ compiler")
    (tmp_path / "program.cpp").write_text(PROGRAM)
    exe = tmp_path / "program"
    subprocess.run([cxx, "-std=c++17", "-O1", "-ffp-contract=off", "-I", CSRC,
                    str(tmp_path / "program.cpp"), "-o", str(exe)], check=True)
    edges = np.arange(1, 8) / 32.0
    xs = np.concatenate([[0.0, 1e-30, np.nextafter(0.25, 0)], edges, np.nextafter(edges, 0),
                         np.random.default_rng(1).uniform(0, 0.25, 100)])
    out = subprocess.run([str(exe)], input="".join(f"{x:.17g}\n" for x in xs),
                         capture_output=True, text=True, check=True).stdout.split()
    for k, x in enumerate(xs):
        for w, n in enumerate((1, 3, 5)):
            e = exact_factor(n, x)
            assert abs(float(out[3 * k + w]) - e) <= 2e-15 * e, (n, x)
