"""A sweep, steps that leave the state in the other population buffer, a restored image and the same sweep again: the
second sweep runs on the restored state, whatever launches an earlier one captured.  Bitwise against a fresh
handle given the same image."""
import numpy as np
import pytest

from paper_1310_7450_gb300 import inputs, lbnlm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("variant", [0, 1])
@pytest.mark.parametrize("prec", ["f64", "f32"])
def test_sweep_runs_on_the_restored_state(prec, variant):
    import torch
    stream = torch.cuda.current_stream().cuda_stream
    nys = [9, 24, 40]
    ps = [dict(inputs.matched_params(0.9, 50.0, 0.1, 1e-3, 1e-5), rho_pert_amp=1e-3, seed=k + 1) for k in range(len(nys))]
    with lbnlm.Channels(4, nys, ps, prec, stream=stream) as a, lbnlm.Channels(4, nys, ps, prec, stream=stream) as b:
        image = np.zeros(lbnlm.lb_state_bytes(a.h), dtype=np.uint8)
        lbnlm.lb_get_state(a.h, image)
        for sim in (a, b):
            lbnlm.lb_sweep_set_config(sim.h, variant, 128, 1)
        a.run_until_steady(-1.0, check_every=10, max_steps=200)
        a.step(1)                                  # the buffers change places
        got = []
        for sim in (a, b):
            lbnlm.lb_set_state(sim.h, image)
            got.append((*sim.run_until_steady(-1.0, check_every=10, max_steps=200), sim.populations()))
    assert np.array_equal(got[0][0], got[1][0]) and np.array_equal(got[0][1], got[1][1])
    for (na, da), (nb, db) in zip(got[0][2], got[1][2]):
        assert np.array_equal(na, nb) and np.array_equal(da, db)
