"""A source that coincides with a target near the origin of coordinates, in a segment
that is wide against delta (needs a GB300).

The box tests of the FP32C kernels hold positions rebuilt from frame-relative ones,
whose rounding grows with the segment's extent; the pair at distance 0 must reach the
FP64 near sum all the same. 32 sources of FP32 coordinates (the frame shifts of the
coincident pair then agree) make one segment of half extent E <= 1.

Bound: 1e-6, the FP32C tolerance, of the pairs' uncancelled values, and for the pairs
beyond delta the shift of the difference by the frame's rounding, four roundings of
E per axis (sqrt(3) 4 2^-24 E), times the kernel's gradient: at most 6 |w f| / (8 pi
r^2) for the Stokeslet and 8 times 6 |w q| / (8 pi r^3) for the stresslet.
"""

import numpy as np
import pytest

import oracle

sk = pytest.importorskip("paper_2310_13908_gb300")
torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("layer", ["single", "double"])
@pytest.mark.parametrize("delta", [1e-10, 1e-9, 3e-9, 1e-8, 1e-6])
def test_coincident_source_in_wide_segment(layer, delta):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    rng = np.random.default_rng(int(-np.log10(delta)))
    d = np.array([delta])
    with sk.Context(0) as c:
        for _ in range(20):
            X = rng.uniform(0.3, 1.0, (32, 3)) * rng.choice([-1.0, 1.0], (32, 3)) + 0.7
            X[11] = rng.uniform(-1, 1, 3) * 10.0 ** rng.uniform(-5, -2)
            X = X.astype(np.float32).astype(np.float64)
            w = rng.uniform(0.5, 1.5, 32)
            f, n = rng.standard_normal((2, 32, 3))
            n /= np.linalg.norm(n, axis=1)[:, None]
            Y = X[11:12]
            E = 0.5 * np.max(np.ptp(X, axis=0))
            r = np.linalg.norm(np.delete(X, 11, 0) - Y, axis=1)
            wf = np.delete(w * np.linalg.norm(f, axis=1), 11) / (8 * np.pi)
            shift = np.sqrt(3) * 4 * 2.0 ** -24 * E
            if layer == "single":
                u = sk.stokes_sl_eval(c.handle, sk.SK_FP32C, sk.SK_HOST, X, w, f, Y, d, 1.0)
                ref = oracle.sl(X, w, f, Y, d, 1.0)
                self_term = oracle.sl(Y, w[11:12], f[11:12], Y, d, 1.0)
                bound = 1e-6 * (np.linalg.norm(self_term) + np.sum(2 * wf / r))
                bound += shift * np.sum(6 * wf / r ** 2)
            else:
                u = sk.stokes_dl_eval(c.handle, sk.SK_FP32C, sk.SK_HOST, X, w, n, f, Y, d)
                ref = oracle.dl(X, w, n, f, Y, d)
                bound = 1e-6 * np.sum(6 * wf / r ** 2) + shift * np.sum(48 * wf / r ** 3)
            assert np.linalg.norm(u - ref) <= bound, X[11]
