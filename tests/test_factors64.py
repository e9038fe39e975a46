"""The FP64 pair kernels' factor table (csrc/sk_factors64.h): s1/rho, s2/rho^3
and s3/rho^5 (Sec. 3.4; reading R7 for s3) as local polynomials in rho^2.

On the CPU the header is compiled with the host compiler and evaluated as the
kernel evaluates it, against 40-digit closed forms. Bound: the FP64 part rounds
a few times (2^-53 each); the FP32 part is at most 2^-24 of the factor (half an
interval is at most 2^-8 (1 + x) wide, and the factor's own scale is 1) and
rounds a few times at 2^-24: together below 1e-14.

On a GPU the pair kernel is compared with the FP64 oracle where its branches
meet: pairs on both sides of rho = 7 (the smoothed range) and rho = 16 (the
table's end), r = 0, and source counts around the chunk, segment and tile edges.
"""

import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2310_13908_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <cstring>
#include <vector>
#include "sk_factors64.h"
using namespace sk;
// stdin: "n x" per line; stdout: the table's value at y = 1 + x rounded to double
int main() {
  std::vector<char> t(F64_TABLES_BYTES);
  f64_build_tables(t.data());
  int n;
  double x;
  while (std::scanf("%d %lf", &n, &x) == 2) {
    const bool dl = n == 5;
    const int f = n == 3, nf = dl ? 1 : 2, tail = dl ? F64_TAIL_DL : F64_TAIL_SL;
    const double* head = (const double*)(t.data() + (dl ? f64_table_bytes(false) : 0));
    const float* tl = (const float*)(head + (size_t)nf * F64_HEAD * F64_N);
    const double y = 1.0 + x;
    uint64_t u;
    std::memcpy(&u, &y, 8);
    const uint32_t hi = (uint32_t)(u >> 32), low = (1u << (20 - F64_SUB_BITS)) - 1;
    const int i = (int)(hi - 0x3ff00000u) >> (20 - F64_SUB_BITS);
    const uint64_t mu = (uint64_t)((hi & ~low) | ((low + 1) >> 1)) << 32;
    double mid;
    std::memcpy(&mid, &mu, 8);
    const double d = y - mid;
    float w = tl[((size_t)f * tail + tail - 1) * F64_N + i];
    for (int k = tail - 2; k >= 0; --k) w = std::fma(w, (float)d, tl[((size_t)f * tail + k) * F64_N + i]);
    const double* c = head + (size_t)f * F64_HEAD * F64_N + i;
    double p = c[3 * F64_N] + (double)(w * (float)d);
    for (int k = 2; k >= 0; --k) p = std::fma(p, d, c[k * F64_N]);
    std::printf("%.17g %.17g\n", y, p);
  }
}
"""


def exact_factor(n, x):
    mp = pytest.importorskip("mpmath").mp
    mp.dps = 120  # the closed forms cancel to rho^5 at small rho
    x = mp.mpf(x)
    if x == 0:
        return {1: mp.mpf(16) / 3, 3: mp.mpf(32) / 3, 5: mp.mpf(128) / 15}[n] / mp.sqrt(mp.pi)
    p = mp.sqrt(x)
    g = mp.exp(-x) / mp.sqrt(mp.pi)
    if n == 1:
        s = mp.erf(p) - mp.mpf(2) / 3 * p * (2 * x - 5) * g
    elif n == 3:
        s = mp.erf(p) - mp.mpf(2) / 3 * p * ((4 * x - 14) * x + 3) * g
    else:
        s = mp.erf(p) - mp.mpf(2) / 9 * p * (((8 * x - 36) * x + 6) * x + 9) * g
    return s / p ** n


def test_table_matches_closed_forms(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("needs a host C++ compiler")
    (tmp_path / "program.cpp").write_text(PROGRAM)
    exe = tmp_path / "program"
    subprocess.run([cxx, "-std=c++17", "-O1", "-ffp-contract=off", "-I", CSRC,
                    str(tmp_path / "program.cpp"), "-o", str(exe)], check=True)
    rng = np.random.default_rng(3)
    edges = [2.0 ** (i // 128) * (1 + (i % 128) / 128) - 1 for i in range(0, 1024, 17)]
    xs = np.concatenate([[0.0, 1e-12, 2.0, 4.84, 49.0, np.nextafter(255.0, 0)], edges[1:],
                         np.nextafter(edges[1:], 0), rng.uniform(0, 12, 150),
                         rng.uniform(0, 255, 60)])
    pts = [(n, x) for n in (1, 3, 5) for x in xs]
    out = subprocess.run([str(exe)], input="".join(f"{n} {x:.17g}\n" for n, x in pts),
                         capture_output=True, text=True, check=True).stdout.split("\n")
    for (n, x), line in zip(pts, out):
        y, v = (float(t) for t in line.split())
        e = exact_factor(n, y - 1.0)  # exact difference: the kernel sees x through y = 1 + x
        assert abs(v - e) <= 1e-14 * e, (n, x)


@pytest.mark.gpu
@pytest.mark.parametrize("layer", ["single", "double"])
@pytest.mark.parametrize("n_src", [1, 7, 8, 9, 33, 127, 129, 1025])
def test_pair_branches_against_oracle(layer, n_src):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import oracle
    import paper_2310_13908_gb300 as sk
    rng = np.random.default_rng(n_src)
    X = 0.3 * rng.standard_normal((n_src, 3))
    w = rng.uniform(0.5, 1.5, n_src) / n_src
    f = rng.standard_normal((n_src, 3))
    nrm = rng.standard_normal((n_src, 3))
    nrm /= np.linalg.norm(nrm, axis=1)[:, None]
    delta = 0.05
    rho = np.array([0.0, 1e-9, 0.3, 2.199, 2.201, 6.999, 7.001, 15.9, 15.99, 16.01, 40.0])
    e = rng.standard_normal((len(rho), 3))
    e /= np.linalg.norm(e, axis=1)[:, None]
    Y = np.concatenate([X[rng.integers(n_src)] + (delta * rho)[:, None] * e,
                        0.5 * rng.standard_normal((70, 3))])
    with sk.Context(0) as c:
        if layer == "single":
            u = sk.stokes_sl_eval(c.handle, sk.SK_FP64, sk.SK_HOST, X, w, f, Y, delta)
            ref = oracle.sl(X, w, f, Y, np.array([delta]), 1.0)
        else:
            u = sk.stokes_dl_eval(c.handle, sk.SK_FP64, sk.SK_HOST, X, w, nrm, f, Y, delta)
            ref = oracle.dl(X, w, nrm, f, Y, np.array([delta]))
    assert np.linalg.norm(u - ref) <= 1e-12 * np.linalg.norm(ref)
    assert np.max(np.abs(u - ref)) <= 1e-12 * np.max(np.abs(ref))
