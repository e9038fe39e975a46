"""Area elements whose square overflows (needs a GB300): W is infinite, as the square
root has it, and not NaN. Tangents of 1.2e77 on a sphere give E G > 1.8e308 near the
equators of the patches."""

import numpy as np
import pytest

import capsule_inputs as ci
from oracle import membrane as mb

sk = pytest.importorskip("paper_2310_13908_gb300")
torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


def test_overflowed_area_element_is_infinite():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    m = 17
    s = ci.make_surface(ci.Sphere(1.0), m)
    X = 1.2e77 * s.X
    with np.errstate(all="ignore"):
        ref = mb.quadrature_weights(m, X)
    with sk.Context(0) as c:
        _, w = sk.membrane_force(c.handle, m, sk.SK_HOST, X, s.X, 2.0, 20.0, weights=True)
    live = s.psi > 0
    assert np.isinf(ref[live]).any() and not np.isnan(ref[live]).any()
    assert np.array_equal(np.isinf(w[live]), np.isinf(ref[live])) and not np.isnan(w[live]).any()
