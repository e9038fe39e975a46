"""Thresholds set anew while requests are on their way (needs a GB300).

A served request takes the thresholds of one moment: whatever sk_set_fp32c_thresholds
does between its preparation and its items, the result is that of the old thresholds or
of the new ones, bit for bit.
"""

import numpy as np
import pytest

import capsule_inputs as ci

sk = pytest.importorskip("paper_2310_13908_gb300")
torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m", [17, 33])
def test_request_keeps_its_thresholds(m):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    s = ci.make_surface(ci.Sphere(1.0), m)
    f = np.random.default_rng(m).standard_normal((s.N, 3))
    args = (s.X, s.w, f, s.X, np.array([2.0 * s.h]))
    kinds = ((0.5, 5.0), (1.0, 6.0))
    with sk.Context(0) as c:
        refs = []
        for k in kinds:
            sk.sk_set_fp32c_thresholds(c.handle, *k)
            refs.append(sk.stokes_sl_eval(c.handle, sk.SK_FP32C, sk.SK_HOST, *args))
        assert not np.array_equal(refs[0], refs[1])
        srv = sk.serve_create(c.handle, max_slots=8)
        try:
            for i in range(100):
                tickets = [sk.serve_submit(srv, *args) for _ in range(4)]
                sk.sk_set_fp32c_thresholds(c.handle, *kinds[i % 2])
                for t in tickets:
                    code, u, _ = sk.serve_poll(srv, t, s.N, timeout_us=30_000_000)
                    assert code == sk.SK_OK
                    assert np.array_equal(u, refs[0]) or np.array_equal(u, refs[1]), i
        finally:
            sk.serve_destroy(srv)
