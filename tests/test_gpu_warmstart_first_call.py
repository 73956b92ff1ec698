"""The first warm-start call of a handle in the middle of a stream capture: it fails (it has tables to upload and waits
for them) and leaves nothing behind that a later call would take for filled.  Later calls equal those of a
handle that saw no capture, bitwise."""
import numpy as np
import pytest

from paper_1310_7450_gb300 import inputs, lbnlm
from stream_capture import Captured

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("first", ["apply", "targets"])
def test_a_failed_first_call_leaves_the_handle_usable(first):
    import torch
    s = torch.cuda.Stream()
    nys = [33, 64, 10]
    ps = [dict(inputs.yield_stress_channel(ny, theta=10.0 * (k + 1), g_x=2e-7 * (64.0 / ny) ** 2)) for k, ny in enumerate(nys)]
    t = [torch.full((len(nys), 768), float("nan"), device="cuda") for _ in range(2)]
    torch.cuda.synchronize()

    def capture(sim):
        def work():
            with pytest.raises(lbnlm.LBError):
                lbnlm.lb_warmstart_apply(sim.h) if first == "apply" else lbnlm.lb_warmstart_targets(sim.h, t[0])
        c = Captured(s.cuda_stream, work)
        assert c.status != 0
        c.close()

    with lbnlm.Channels(4, nys, ps, "f64", stream=s.cuda_stream) as a, lbnlm.Channels(4, nys, ps, "f64", stream=s.cuda_stream) as b:
        capture(a)
        for sim, targets in zip((a, b), t):
            lbnlm.lb_warmstart_apply(sim.h)
            sim.step(3)
            lbnlm.lb_warmstart_targets(sim.h, targets)
        for (na, da), (nb, db) in zip(a.populations(), b.populations()):
            assert np.array_equal(na, nb) and np.array_equal(da, db)
        torch.cuda.synchronize()
        assert torch.isfinite(t[0]).all() and torch.equal(t[0], t[1])
