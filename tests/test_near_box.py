"""The box tests of the FP32 pair kernels (csrc/sk_near_box.h), compiled with the host
compiler: no pair whose FP32 difference lies inside rho_c delta may be cleared, and no
source that lies well outside may be kept. Segments of 32 sources of any extent and
offset, targets at or beside one of them, delta down to 1e-10 of the extent."""

import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2310_13908_gb300", "csrc")

# per draw: 32 sources, one target, delta on stdin; out: pairs inside by the kernel's FP32
# difference, of those the ones cleared by the segment's and by the source's test, and
# sources kept at more than twice the reach
PROGRAM = r"""
#include <cstdio>
#include "sk_near_box.h"
using namespace sk::p32;
static float mid(float lo, float hi) { return (lo + hi) * 0.5f; }
int main() {
  double y[32][3], x[3], delta;
  for (;;) {
    for (auto& p : y)
      if (std::scanf("%lf %lf %lf", p, p + 1, p + 2) != 3) return 0;
    if (std::scanf("%lf %lf %lf %lf", x, x + 1, x + 2, &delta) != 4) return 1;
    float lo[3], hi[3], c[3], xh[3], xl[3], t[3], cmax = 0.f;
    for (int a = 0; a < 3; ++a) {
      lo[a] = 3e38f, hi[a] = -3e38f;
      for (auto& p : y) lo[a] = std::fmin(lo[a], (float)p[a]), hi[a] = std::fmax(hi[a], (float)p[a]);
      c[a] = mid(lo[a], hi[a]);
      xh[a] = (float)x[a], xl[a] = (float)(x[a] - (double)xh[a]);
      t[a] = (xh[a] - c[a]) + xl[a];
      cmax = std::fmax(cmax, std::fabs(xh[a]));
    }
    const float rc2 = (float)((5.0 * delta) * (5.0 * delta)), rc = std::sqrt(rc2);
    const float rm = rc * 1.00005f + box_margin(cmax, rc);
    const NearBox box{{xh[0], xh[1], xh[2]}, {xh[0], xh[1], xh[2]}, rm * rm};
    const bool seg = box.reaches(segment_span(lo[0], hi[0]), segment_span(lo[1], hi[1]),
                                 segment_span(lo[2], hi[2]));
    int inside = 0, by_segment = 0, by_source = 0, kept = 0;
    for (auto& p : y) {
      float r[3], d[3];
      double far2 = 0.0;
      for (int a = 0; a < 3; ++a) {
        r[a] = -(float)(p[a] - (double)c[a]);
        d[a] = t[a] + r[a];
        far2 += (x[a] - p[a]) * (x[a] - p[a]);
      }
      const float r2 = d[2] * d[2] + (d[1] * d[1] + d[0] * d[0]);
      const bool src = box.reaches(source_span(c[0], r[0]), source_span(c[1], r[1]),
                                   source_span(c[2], r[2]));
      if (r2 < rc2) ++inside, by_segment += !seg, by_source += !src;
      const double ext = std::fmax(hi[0] - lo[0], std::fmax(hi[1] - lo[1], hi[2] - lo[2]));
      const double reach = 5.0 * delta + 2e-6 * (cmax + ext);
      kept += src && std::sqrt(far2) > 2.0 * reach;
    }
    std::printf("%d %d %d %d\n", inside, by_segment, by_source, kept);
  }
}
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("needs a host C++ compiler")
    d = tmp_path_factory.mktemp("near_box")
    (d / "program.cpp").write_text(PROGRAM)
    subprocess.run([cxx, "-std=c++17", "-O1", "-ffp-contract=off", "-I", CSRC,
                    str(d / "program.cpp"), "-o", str(d / "program")], check=True)

    def go(draws):
        text = "\n".join(" ".join(repr(float(v)) for v in q) for q in draws)
        out = subprocess.run([str(d / "program")], input=text, capture_output=True, text=True,
                             check=True).stdout
        return np.array([[int(v) for v in row.split()] for row in out.splitlines()])

    return go


@pytest.mark.parametrize("offset", [0.0, 1e-3, 1.0, 1e3])
@pytest.mark.parametrize("delta", [1e-10, 1e-9, 3e-9, 1e-8, 1e-7, 1e-5, 1e-2])
def test_no_near_pair_is_cleared(run, offset, delta):
    rng = np.random.default_rng(int(1e4 * offset) + int(-np.log10(delta)))
    draws = []
    for k in range(400):
        Y = rng.uniform(0.0, 1.0, (32, 3)) * 10.0 ** rng.uniform(-3, 0) + offset
        j = rng.integers(32)
        if k % 2:  # a target near the origin of coordinates, which the margin scales with
            Y[j] = rng.uniform(-1, 1, 3) * 10.0 ** rng.uniform(-8, -2)
        x = Y[j] + (k % 4 > 1) * delta * rng.standard_normal(3)
        draws.append(np.concatenate([Y.ravel(), x, [delta]]))
    inside, by_segment, by_source, kept = run(draws).sum(0)
    assert inside > 0
    assert by_segment == 0 and by_source == 0 and kept == 0
