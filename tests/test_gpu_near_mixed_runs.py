"""Near runs of every length in one group's list (needs a GB300).

Each target's part of its group's near list is ranked by a warp up to 32 and up to 128
entries, and sorted by one lane beyond. One delta for all targets cannot reach the last
without overflowing the list (96 entries a target on average), so a fifth of the targets
gets a delta of 4h to 8h and the others 2h: runs of 2 to over 200. The counted pairs are
those of the CPU, up to pairs within FP32 rounding of the limit; the sums match the
oracle at the tolerance of the parity tests.
"""

import numpy as np
import pytest

import capsule_inputs as ci
import oracle

sk = pytest.importorskip("paper_2310_13908_gb300")
torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu
RHO_T = 0.5


@pytest.mark.parametrize("layer", ["single", "double"])
def test_mixed_near_runs(layer):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    rng = np.random.default_rng(19)
    s = ci.make_surface(ci.Sphere(1.0), 33)
    f = rng.standard_normal((s.N, 3)) + np.array([1.0, 0.0, 0.0])
    ratio = np.where(rng.random(s.N) < 0.2, rng.uniform(4.0, 8.0, s.N), 2.0)
    delta = ratio * s.h
    X = s.X[s.w != 0]
    runs, edge = np.zeros(s.N, dtype=int), 0
    for i, y in enumerate(s.X):
        rho = np.linalg.norm(X - y, axis=1) / delta[i]
        runs[i] = np.count_nonzero(rho < RHO_T)
        edge += np.count_nonzero(np.abs(rho / RHO_T - 1.0) < 1e-6)
    assert runs.min() < 32 and runs.max() > 128 and np.any((runs > 32) & (runs <= 128))
    with sk.Context(0) as c:
        if layer == "single":
            u = sk.stokes_sl_eval(c.handle, sk.SK_FP32C, sk.SK_HOST, s.X, s.w, f, s.X, delta)
            ref = oracle.sl(s.X, s.w, f, s.X, delta, 1.0)
        else:
            u = sk.stokes_dl_eval(c.handle, sk.SK_FP32C, sk.SK_HOST, s.X, s.w, s.n, f, s.X, delta)
            ref = oracle.dl(s.X, s.w, s.n, f, s.X, delta)
        st = sk.sk_last_eval_stats(c.handle)
    assert st["overflow_targets"] == 0
    assert abs(st["near_pairs"] - runs.sum()) <= edge
    assert np.linalg.norm(u - ref) <= 1e-6 * np.linalg.norm(ref)
