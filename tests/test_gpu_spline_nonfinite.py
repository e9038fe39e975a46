"""A node value that is not finite reaches its whole grid lines (needs a GB300).

The spline solves couple every term of a line, so one such node makes every spline value
of its patch not finite, and with them the derivatives of each node whose stencil or
blend takes one. Lines of 40 and 96 nodes lie within and beyond the runs that a lane's
entering value is taken from. The oracle's pattern is the reference; its stencil
multiplies the node itself by 0, which the kernel's leaves out, so that node may differ.
"""

import numpy as np
import pytest

from oracle import membrane as mb

sk = pytest.importorskip("paper_2310_13908_gb300")
torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m", [41, 97])
@pytest.mark.parametrize("at", [0.5, 0.1])
def test_nonfinite_reaches_whole_lines(m, at):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    n = m - 1
    g = np.random.default_rng(m).standard_normal((6 * n * n, 4))
    node = 2 * n * n + int(at * n) * n + int((1 - at) * n)
    g[node, :3] = np.nan, np.inf, -np.inf
    with np.errstate(invalid="ignore"):
        ref_u, ref_v = mb.surface_derivatives(m, g)
    with sk.Context(0) as c:
        gu, gv = sk.surface_derivatives(c.handle, m, sk.SK_HOST, g)
    for a, b in ((gu, ref_u), (gv, ref_v)):
        lost = np.isfinite(a) & ~np.isfinite(b)
        lost[node] = False
        assert not lost.any(), lost.sum(0)
        assert np.max(np.abs(a[:, 3] - b[:, 3])) <= 1e-11 * np.max(np.abs(b[:, 3]))
