"""Spline slope solves at the edges of their split into lane runs (needs a GB300).

A grid line of n = m - 1 nodes is solved by 16 lanes, each with a run of
ceil((n - 2) / 16) terms: lines with one term per lane, with empty lanes, with
a ragged last run, and longer ones. The
derivatives of random node values (no smooth field hides an end condition) are
compared with the oracle's at the bound of the derivative parity tests, 1e-11 of
the largest value; field counts cover one, a group of three, and a ragged group.
"""

import numpy as np
import pytest

from oracle import membrane as mb

sk = pytest.importorskip("paper_2310_13908_gb300")
torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,n_fields", [(6, 1), (7, 4), (10, 3), (18, 2), (19, 3), (20, 1),
                                        (35, 5), (161, 1), (162, 1)])
def test_slope_runs_match_oracle(m, n_fields):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    g = np.random.default_rng(m).standard_normal((6 * (m - 1) ** 2, n_fields))
    ref_u, ref_v = mb.surface_derivatives(m, g)
    with sk.Context(0) as c:
        gu, gv = sk.surface_derivatives(c.handle, m, sk.SK_HOST, g)
    for a, b in ((gu, ref_u), (gv, ref_v)):
        assert np.max(np.abs(a - b)) <= 1e-11 * np.max(np.abs(b))
