"""The single-block sort against the multi-launch sorts, bit for bit (needs a GB300).

Three contexts order the same points: the default one (a single block up to 1024 points),
one with the single block up to 2^24 points (SK_SMALL_SORT_POINTS) and one without it.
The stable order, and with it every result, is the same. Sizes: edges of a block's tiles
of 256 and 1024 keys, several tiles in one block, the default's limit, and 131,072 |
131,073, where the number of passes changes.
"""

import os

import numpy as np
import pytest

sk = pytest.importorskip("paper_2310_13908_gb300")
torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def contexts():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    old = os.environ.get("SK_SMALL_SORT_POINTS")
    out = [sk.Context(0)]
    try:
        for points in (1 << 24, 0):
            os.environ["SK_SMALL_SORT_POINTS"] = str(points)
            out.append(sk.Context(0))
    finally:
        if old is None:
            os.environ.pop("SK_SMALL_SORT_POINTS", None)
        else:
            os.environ["SK_SMALL_SORT_POINTS"] = old
    yield out
    for c in out:
        c.close()


@pytest.mark.parametrize("n", [1, 2, 255, 256, 257, 1023, 1024, 1025, 2047, 2049, 8192, 32769,
                               131072, 131073])
@pytest.mark.parametrize("prec", [sk.SK_FP64, sk.SK_FP32C], ids=["fp64", "fp32c"])
def test_sorts_agree(contexts, n, prec):
    rng = np.random.default_rng(n)
    X = rng.standard_normal((n, 3))
    X[: n // 3] = X[rng.integers(0, n, n // 3)]  # equal keys: the order must be stable
    w = rng.uniform(0.5, 1.5, n)
    w[rng.random(n) < 0.2] = 0.0
    f = rng.standard_normal((n, 3))
    few = rng.standard_normal((70, 3))
    both = []
    for c in contexts:
        u = sk.stokes_sl_eval(c.handle, prec, sk.SK_HOST, X, w, f, few, 0.05)
        v = sk.stokes_sl_eval(c.handle, prec, sk.SK_HOST, few, np.ones(70), few, X, 0.05)
        both.append((u, v))
    for u, v in both[1:]:
        assert np.array_equal(u, both[0][0]) and np.array_equal(v, both[0][1])
