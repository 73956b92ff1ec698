"""The boundary columns' means of pressure-driven channels at heights on both sides of a block of rows and of as many
blocks as a block has threads, in one handle: two steps from random states against the FP64 oracle, to the
bound that the other pressure-driven tests hold after 40."""
import numpy as np
import pytest

import oracle
from paper_1310_7450_gb300 import inputs, lbnlm

pytestmark = pytest.mark.gpu


def test_heights_around_the_blocks():
    import torch
    oracle.build()
    nx, nys, amp = 3, [3, 255, 256, 257, 513, 65536, 65537], 1e-2
    p = inputs.matched_params(0.9, 10.0, 0.1, 1e-3, 1e-4)
    w = oracle.equilibrium(1.0, 0.0, 0.0)
    states = []
    for k, ny in enumerate(nys):
        rng = np.random.default_rng(900 + k)
        st = oracle.init_state(1.0 + amp * rng.uniform(-1, 1, (ny, nx)))
        st.dev += amp * rng.uniform(-1, 1, st.dev.shape) * w[:, None, None]
        states.append(st)
    with lbnlm.Channels(nx, nys, [p] * len(nys), "f64", stream=torch.cuda.current_stream().cuda_stream, x_mode="gpbc") as sim:
        sim.set_populations([st.nstar for st in states], [st.drho for st in states])
        sim.step(2)
        got = sim.populations()
    for (n, _), st in zip(got, states):
        oracle.run(dict(p, x_mode="gpbc"), st, 2)
        assert np.abs(n - st.nstar).max() < 1e-14 * np.abs(st.nstar).max()
