"""Stochastic rounding in the row march where a value is an infinity or a NaN: the node that pulls it is stored
as such, and the other nodes of its row and strip bitwise as without it (even and odd widths).  Only that
strip's row is compared: work that starts after a node was found unstable is not done."""
import numpy as np
import pytest

from paper_1310_7450_gb300 import inputs, lbnlm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bad", [np.inf, np.nan])
@pytest.mark.parametrize("nx,ny", [(256, 1030), (257, 1031)])
def test_nonfinite_value_is_stored_and_spoils_no_other(nx, ny, bad):
    import torch
    p = dict(inputs.matched_params(0.9, 100.0, 0.1, 1e-3, 1e-5), rho_pert_amp=1e-2, seed=nx)
    y, out = ny // 2, []
    for v in (None, bad):
        with lbnlm.Channels(nx, ny, p, "bf16", flags=lbnlm.LB_GRID_BF16_STOCHASTIC,
                            stream=torch.cuda.current_stream().cuda_stream) as sim:
            assert lbnlm.lb_uses_row_march(sim.h)
            n, d = sim.populations()[0]
            if v is not None:
                n[3, y, 7] = v   # moves with c_x = -1: pulled by the node at x = 6
            lbnlm.lb_set_populations(sim.h, n.ravel(), d.ravel(), None)
            lbnlm.lb_step(sim.h, 1)
            out.append(sim.populations()[0][0][:, y])
    good, spoilt = out
    assert np.isfinite(good).all() and not np.isfinite(spoilt[:, 6]).all()
    assert np.array_equal(good[:, 12:80], spoilt[:, 12:80])
