"""A small channel that becomes unstable in the middle of a run of on-chip steps: what is read back afterwards is the
state it stopped in, however many further calls (which do nothing) lie in between."""
import numpy as np
import pytest

from paper_1310_7450_gb300 import inputs, lbnlm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,kw", [("f64", {}), ("f32", {}), ("bf16", {}), ("f32", dict(stress_mode=1))])
def test_the_stopped_state_stays(prec, kw):
    import torch
    p = dict(inputs.matched_params(0.9, 10.0, 0.1, 1e-3, 3e-3), rho_pert_amp=0.0)   # |u| passes 0.3 after ~100 steps
    with lbnlm.Channels(4, 64, p, prec, stream=torch.cuda.current_stream().cuda_stream, **kw) as sim:
        sim.step(2000)
        assert list(sim.status()) == [1]
        n, d = sim.populations()[0]
        assert np.abs(n[1] - n[3]).max() > 0.1                     # (moving: not the state of rest)
        for more in (1, 3, 2, 40, 1):
            assert sim.step(more) == lbnlm.LB_EUNSTABLE
            m, e = sim.populations()[0]
            assert np.array_equal(n, m) and np.array_equal(d, e)
