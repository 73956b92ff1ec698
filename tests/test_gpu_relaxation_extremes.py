"""The relaxation-time extensions where tau(rho) leaves the range of normal numbers (a reference density far from the
fluid's): infinite (the fluidity is then the shear rate's alone), zero, and among the subnormal numbers.  FP64 random states against the oracle, to the bounds of the other relaxation-model tests."""
import numpy as np
import pytest

import oracle
from paper_1310_7450_gb300 import inputs, lbnlm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("beta,tau_f", [(2.0, 25.0), (-2.0, 25.0), (-2.0, 0.0), (-0.7193, 0.0)])
@pytest.mark.parametrize("mode", [0, 1])
def test_extreme_relaxation_times(beta, tau_f, mode):
    import torch
    oracle.build()
    nx, ny, amp = 40, 13, 1e-2
    p = dict(inputs.matched_params(0.9, 10.0, 0.1, 1e-3, 1e-5), beta_rho=beta, rho_ref=1e-3, tau_f=tau_f, stress_mode=mode)
    rng = np.random.default_rng(7)
    st = oracle.init_state(1.0 + amp * rng.uniform(-1, 1, (ny, nx)))
    st.dev += amp * rng.uniform(-1, 1, st.dev.shape) * oracle.equilibrium(1.0, 0.0, 0.0)[:, None, None]
    with lbnlm.Channels(nx, ny, p, "f64", stress_mode=mode, flags=lbnlm.LB_GRID_RELAXATION_MODEL,
                        stream=torch.cuda.current_stream().cuda_stream) as sim:
        lbnlm.lb_set_relaxation_model(sim.h, -1, beta, 1e-3, tau_f)
        sim.set_populations([st.nstar], [st.drho], [np.zeros((3, ny, nx))] if mode else None)
        sim.step(5)
        assert list(sim.status()) == [0]
        (u_g, s_g, r_g), = sim.fields()
    oracle.run(p, st, 5)
    u_o, s_o, r_o = oracle.fields(p, st)
    assert np.all(np.isfinite(u_o)) and np.all(np.isfinite(s_o))
    assert np.abs(u_g - u_o).max() <= 1e-12 * np.abs(u_o).max()
    assert np.abs(s_g - s_o).max() <= 1e-11 * max(np.abs(s_o).max(), 1e-3 * np.abs(u_o).max())
    assert np.abs(r_g - r_o).max() < 1e-13
