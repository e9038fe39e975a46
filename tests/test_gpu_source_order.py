"""The packed sources' order at the edges of its pattern (needs a GB300).

Segments of 32 sources are dealt out to tiles of 8 (SK_FP32C) and to strides of 16
(SK_FP64); remainders stay in place. A source that was lost or packed twice would
change a sum: random sources, a fifth more of them without weight, against the FP64
oracle at the tolerances of the parity tests.
"""

import numpy as np
import pytest

import oracle

sk = pytest.importorskip("paper_2310_13908_gb300")
torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu
TOL = {sk.SK_FP64: 1e-12, sk.SK_FP32C: 1e-6}


@pytest.mark.parametrize("n", [1, 31, 33, 255, 256, 257, 511, 512, 513, 543, 545, 1025, 2047, 2305])
@pytest.mark.parametrize("prec", [sk.SK_FP64, sk.SK_FP32C], ids=["fp64", "fp32c"])
def test_every_source_is_packed_once(n, prec):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    rng = np.random.default_rng(n)
    total = n + (n + 4) // 5
    X = rng.standard_normal((total, 3))
    w = rng.uniform(0.5, 1.5, total) / n
    w[rng.permutation(total)[n:]] = 0.0
    f = rng.standard_normal((total, 3)) + np.array([1.0, 0.0, 0.0])
    Y = rng.standard_normal((70, 3))
    with sk.Context(0) as c:
        u = sk.stokes_sl_eval(c.handle, prec, sk.SK_HOST, X, w, f, Y, 0.1)
    ref = oracle.sl(X, w, f, Y, np.array([0.1]), 1.0)
    assert np.linalg.norm(u - ref) <= TOL[prec] * np.linalg.norm(ref)
