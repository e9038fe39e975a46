"""Items that follow a block finish on the same CTA of the server (needs a GB300).

The finish of a target block sorts its near lists in the shared memory of the source
stages, which the CTA's next item fills by bulk copies. Wide delta gives long lists;
with more items than CTAs every CTA takes several. Served results equal the standalone
ones bit for bit, round after round.
"""

import numpy as np
import pytest

import capsule_inputs as ci

sk = pytest.importorskip("paper_2310_13908_gb300")
torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ratio", [2.0, 4.0])
def test_items_after_a_finish(ratio):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    rng = np.random.default_rng(int(ratio))
    reqs = []
    for m in (9, 17, 17, 25, 33, 41):
        s = ci.make_surface(ci.Sphere(1.0), m)
        reqs.append((s.X, s.w, rng.standard_normal((s.N, 3)), s.X, np.array([ratio * s.h])))
    with sk.Context(0) as c:
        refs = [sk.stokes_sl_eval(c.handle, sk.SK_FP32C, sk.SK_HOST, *r) for r in reqs]
        srv = sk.serve_create(c.handle, max_slots=8)
        try:
            for _ in range(10):
                tickets = [sk.serve_submit(srv, *r) for r in reqs]
                for t, r, ref in zip(tickets, reqs, refs):
                    code, u, _ = sk.serve_poll(srv, t, r[3].shape[0], timeout_us=30_000_000)
                    assert code == sk.SK_OK and np.array_equal(u, ref)
        finally:
            sk.serve_destroy(srv)
