"""FP64 steps of a fluid with a vanishing critical strain: the Maxwell time falls to nothing wherever there is shear,
and stays tau where there is none.  Random states, and rest, against the oracle, to the bounds of the other FP64
parity tests."""
import numpy as np
import pytest

import oracle
from paper_1310_7450_gb300 import inputs, lbnlm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("gamma_c", [3e-307, 1e-300, 1e-200, 1e-20])
@pytest.mark.parametrize("rest", [False, True])
def test_steps_match_the_oracle(gamma_c, rest):
    import torch
    oracle.build()
    nx, ny, amp = 6, 20, 1e-2
    p = dict(inputs.matched_params(0.9, 50.0, 0.1, 1e-3, 0.0 if rest else 1e-5), gamma_c=gamma_c)
    st = oracle.init_state(np.ones((ny, nx)))
    if not rest:
        rng = np.random.default_rng(3)
        st.dev += amp * rng.uniform(-1, 1, st.dev.shape) * oracle.equilibrium(1.0, 0.0, 0.0)[:, None, None]
    with lbnlm.Channels(nx, ny, p, "f64", stream=torch.cuda.current_stream().cuda_stream) as sim:
        sim.set_populations([st.nstar], [st.drho])
        sim.step(12)
        assert list(sim.status()) == [0]
        (n, d), = sim.populations()
        (u, s, r), = sim.fields()
    oracle.run(p, st, 12)
    u_o, s_o, r_o = oracle.fields(p, st)
    assert np.abs(n - st.nstar).max() < 1e-14 and np.abs(r - r_o).max() < 1e-14
    assert np.abs(u - u_o).max() <= 1e-12 * max(np.abs(u_o).max(), 1e-3)
    assert np.abs(s - s_o).max() <= 1e-11 * max(np.abs(s_o).max(), 1e-6)
