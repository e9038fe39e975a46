"""Lengths beyond the place of the padding sources (needs a GB300).

Packed sources are padded with sources without density 1e15 away. Scaled by 2^53 = 9e15
a sphere's delta exceeds that, so padding lies inside rho_T delta of its targets; it must
not enter the near lists. Scaling by a power of two scales the single layer by its
inverse: the results are compared with those at scale 1, within the FP32C tolerance
(only the order of the sort and the margins may differ).
"""

import numpy as np
import pytest

import capsule_inputs as ci

sk = pytest.importorskip("paper_2310_13908_gb300")
torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu
SCALE = 2.0 ** 53


@pytest.mark.parametrize("path", ["eval", "fmm", "serve"])
@pytest.mark.parametrize("m", [9, 12, 18])
def test_padding_is_never_listed(path, m):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    s = ci.make_surface(ci.Ellipsoid(1.0, 0.8, 0.6), m)
    f = np.random.default_rng(m).standard_normal((s.N, 3))
    delta = np.array([2.0 * s.h])

    def run(c, X, d):
        if path == "eval":
            return sk.stokes_sl_eval(c.handle, sk.SK_FP32C, sk.SK_HOST, X, s.w, f, X, d, 1.0)
        if path == "fmm":
            sk.sk_set_fp32c_thresholds(c.handle, 2.0, 8.0)
            return sk.stokes_sl_eval_fmm(c.handle, sk.SK_HOST, X, s.w, f, X, d, 1.0, X[:: s.N // 8][:8],
                                         4, 4, precision=sk.SK_FP32C)
        srv = sk.serve_create(c.handle, max_slots=2)
        try:
            t = sk.serve_submit(srv, X, s.w, f, X, d, 1.0)
            code, u, _ = sk.serve_poll(srv, t, s.N, timeout_us=30_000_000)
            assert code == sk.SK_OK
            return u
        finally:
            sk.serve_destroy(srv)

    with sk.Context(0) as c:
        a, b = run(c, s.X, delta), SCALE * run(c, SCALE * s.X, SCALE * delta)
    assert np.linalg.norm(b - a) <= 1e-6 * np.linalg.norm(a)
