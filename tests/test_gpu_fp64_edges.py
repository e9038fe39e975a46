"""FP64 building blocks and sums at the ends of the number range (needs a GB300).

The reciprocal roots, reciprocals and conversions that csrc/sk_internal.h puts in the
place of library calls, compiled into a program of their own and run over random
mantissas at every exponent and over edge values. Bounds, from the roundings named
there: |y sqrt(x) - 1| <= 2^-53 + 2^-54 + 2^-58 for the root and |y x - 1| <= 2^-53 +
2^-58 for the reciprocal, taken in long double; edge values and arguments outside the
fast range as the library gives them; conversions exactly. Then FP64 sums whose squared
distances are subnormal.
"""

import os
import shutil
import subprocess

import numpy as np
import pytest

import oracle

sk = pytest.importorskip("paper_2310_13908_gb300")
torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu
CSRC = os.path.join(os.path.dirname(os.path.abspath(sk.__file__)), "csrc")

PROGRAM = r"""
#include <cstdio>
#include <vector>
#include "sk_internal.h"
__global__ void k(const double* x, double* out, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  double* o = out + 6 * (size_t)i;
  o[0] = sk::rsqrt_fp64(x[i]);
  o[1] = rsqrt(x[i]);
  o[2] = sk::rcp_fp64(x[i]);
  o[3] = 1.0 / x[i];
  const bool fits = fabs(x[i]) < 3e38;
  o[4] = fits ? (double)sk::narrow(x[i]) : 0.0;
  o[5] = sk::widen(__double2float_rn(x[i]));
}
int main(int, char** v) {
  std::vector<double> x;
  FILE* f = std::fopen(v[1], "rb");
  for (double t; std::fread(&t, 8, 1, f) == 1;) x.push_back(t);
  std::fclose(f);
  const int n = (int)x.size();
  std::vector<double> out(6 * x.size());
  double *dx, *dout;
  if (cudaMalloc(&dx, 8 * x.size()) || cudaMalloc(&dout, 48 * x.size())) return 1;
  cudaMemcpy(dx, x.data(), 8 * x.size(), cudaMemcpyHostToDevice);
  k<<<(n + 255) / 256, 256>>>(dx, dout, n);
  if (cudaMemcpy(out.data(), dout, 48 * x.size(), cudaMemcpyDeviceToHost)) return 1;
  f = std::fopen(v[2], "wb");
  std::fwrite(out.data(), 8, out.size(), f);
  return std::fclose(f);
}
"""


@pytest.fixture(scope="module")
def device(tmp_path_factory):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("needs nvcc")
    d = tmp_path_factory.mktemp("fp64")
    (d / "program.cu").write_text(PROGRAM)
    subprocess.run([nvcc, "-std=c++17", "-O3", "-gencode", "arch=compute_103a,code=sm_103a",
                    "--expt-relaxed-constexpr", "-I", CSRC, str(d / "program.cu"), "-o",
                    str(d / "program")], check=True)

    def run(x):
        x.tofile(d / "in")
        subprocess.run([str(d / "program"), str(d / "in"), str(d / "out")], check=True)
        return np.fromfile(d / "out").reshape(-1, 6)

    return run


def test_reciprocals_and_conversions(device):
    rng = np.random.default_rng(5)
    e = np.repeat(np.arange(-1074, 1024), 200)
    with np.errstate(all="ignore"):
        x = np.ldexp(1.0 + rng.random(e.size), e)
        x = x[np.isfinite(x)]
    edges = np.array([0.0, 5e-324, 2.0 ** -1022, np.nextafter(2.0 ** -1022, 0), 2.0 ** 1021,
                      np.nextafter(2.0 ** 1021, 0), np.finfo(float).max, np.inf, np.nan])
    x = np.concatenate([x, edges, -x[::50], -edges])
    o = device(x)
    normal = (np.abs(x) >= 2.0 ** -1022) & np.isfinite(x)
    root = normal & (x > 0)
    xl = x.astype(np.longdouble)
    # 2^-53 + 2^-54 + 2^-58 with the squaring done exactly enough: (y^2 x - 1) / 2
    y = o[:, 0].astype(np.longdouble)
    s = np.ldexp(xl[root], -2 * (np.frexp(x[root])[1] // 2))
    t = np.ldexp(y[root], np.frexp(x[root])[1] // 2)
    assert np.max(np.abs((t * t * s - 1) / 2)) <= 2.0 ** -53 + 2.0 ** -54 + 2.0 ** -58
    assert np.array_equal(o[~root, 0], o[~root, 1], equal_nan=True)
    fast = (x >= 2.0 ** -1022) & (x < 2.0 ** 1021)
    y = o[:, 2].astype(np.longdouble)
    assert np.max(np.abs(y[fast] * xl[fast] - 1)) <= 2.0 ** -53 + 2.0 ** -58
    assert np.array_equal(o[~fast, 2], o[~fast, 3], equal_nan=True)
    with np.errstate(all="ignore"):
        f = x.astype(np.float32)
        back = f.astype(np.float64)
        toward0 = np.where(np.abs(back) > np.abs(x), np.nextafter(f, np.float32(0)), f)
    assert np.array_equal(o[:, 5], back, equal_nan=True)
    fits = np.abs(x) < 3e38
    want = np.where(np.abs(x) < 2.0 ** -126, 0.0, toward0.astype(np.float64))
    assert np.array_equal(o[fits, 4], want[fits])


@pytest.mark.parametrize("near", [False, True])
def test_subnormal_squared_distances(near):
    """Distances in (1, 2) 2^-512, whose squares are subnormal, by the far loop, and, with a
    target at unit distance in the same warp, by the near loop at a delta of 2^-516. The
    single layer scales with the inverse of the lengths; a square is off by at most 3 2^-1075
    of 2^-1024, 1/r^3 by 4.5 2^-51."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    rng = np.random.default_rng(int(near))
    lam = 2.0 ** -512
    dirs = rng.standard_normal((40, 3))
    X = dirs / np.linalg.norm(dirs, axis=1)[:, None] * rng.uniform(1.05, 1.9, (40, 1))
    w, f = rng.uniform(0.5, 1.5, 40), rng.standard_normal((40, 3))
    Y, d = np.zeros((1, 3)), np.array([2.0 ** -4])
    ref = oracle.sl(X, w, f, Y, d, 1.0)
    Yl = np.concatenate([Y, [[1.0, 1.0, 1.0]]]) if near else Y
    with sk.Context(0) as c:
        u = sk.stokes_sl_eval(c.handle, sk.SK_FP64, sk.SK_HOST, lam * X, w, f, Yl, lam * d, 1.0)
    assert np.linalg.norm(lam * u[0] - ref[0]) <= 1e-12 * np.linalg.norm(ref)
