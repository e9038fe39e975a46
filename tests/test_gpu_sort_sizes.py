"""The spatial sorts at the edges of their launch plans (needs a GB300).

Point sets of up to 32,768 / 65,536 / 131,072 points are sorted with 1, 2 or 4
points per thread and tile counts in one array; larger ones take another plan. A
sort that lost, repeated or misplaced a point would change a sum: random sources
with random weights (a fifth of them zero), a handful of targets, against the
FP64 oracle at the tolerances of the parity tests; then as many targets from a
handful of sources, where every target must get its own value.
"""

import numpy as np
import pytest

import oracle

sk = pytest.importorskip("paper_2310_13908_gb300")
torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu
TOL = {sk.SK_FP64: 1e-12, sk.SK_FP32C: 1e-6}


@pytest.mark.parametrize("n", [3073, 32768, 32769, 65536, 65537, 131072, 131073])
@pytest.mark.parametrize("prec", [sk.SK_FP64, sk.SK_FP32C], ids=["fp64", "fp32c"])
def test_sort_plan_edges(n, prec):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    rng = np.random.default_rng(n)
    X = rng.standard_normal((n, 3))
    w = rng.uniform(0.5, 1.5, n) / n
    w[rng.random(n) < 0.2] = 0.0
    f = rng.standard_normal((n, 3)) + np.array([1.0, 0.0, 0.0])
    few = 40
    delta = 0.02
    with sk.Context(0) as c:
        u = sk.stokes_sl_eval(c.handle, prec, sk.SK_HOST, X, w, f, X[:few], delta)
        v = sk.stokes_sl_eval(c.handle, prec, sk.SK_HOST, X[:few], w[:few], f[:few], X, delta)
    ref = oracle.sl(X, w, f, X[:few], np.array([delta]), 1.0)
    assert np.linalg.norm(u - ref) <= TOL[prec] * np.linalg.norm(ref)
    ref = oracle.sl(X[:few], w[:few], f[:few], X, np.array([delta]), 1.0)
    assert np.linalg.norm(v - ref) <= TOL[prec] * np.linalg.norm(ref)
    assert np.max(np.abs(v - ref)) <= 10 * TOL[prec] * np.max(np.abs(ref))
