"""Near sums of targets with about 15 to 100 near pairs each (needs a GB300).

Runs of up to 32, 33 to 128 and more entries of a group's near list are sorted in
three ways; delta from 2h to 5h takes a target through them. Against the FP64 oracle
at the tolerance of the parity tests.
"""

import numpy as np
import pytest

import capsule_inputs as ci
import oracle

sk = pytest.importorskip("paper_2310_13908_gb300")
torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ratio", [2, 3, 4, 5])
def test_near_runs_match_oracle(ratio):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    s = ci.make_surface(ci.Sphere(1.0), 33)
    f = np.random.default_rng(ratio).standard_normal((s.N, 3)) + np.array([1.0, 0.0, 0.0])
    delta = np.array([ratio * s.h])
    with sk.Context(0) as c:
        u = sk.stokes_sl_eval(c.handle, sk.SK_FP32C, sk.SK_HOST, s.X, s.w, f, s.X, delta)
    ref = oracle.sl(s.X, s.w, f, s.X, delta, 1.0)
    assert np.linalg.norm(u - ref) <= 1e-6 * np.linalg.norm(ref)
