"""lb_warmstart_apply for fluids with a vanishing critical strain (the argument of the closed form's square root is then 0
or subnormal in the middle of the channel) and a large one, against lb_set_fields with the reference profiles, to
the bound of the other warm-start tests."""
import numpy as np
import pytest

import warmstart_reference as ref
from paper_1310_7450_gb300 import inputs, lbnlm, warmstart

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("gamma_c", [1e-300, 1e-200, 1e-155, 1e-100, 1e-6, 10.0])
def test_start_state_equals_set_fields(gamma_c):
    import torch
    stream = torch.cuda.current_stream().cuda_stream
    nys = [3, 33, 64]
    ps = [dict(inputs.yield_stress_channel(ny, theta=10.0, g_x=2e-7 * (64.0 / ny) ** 2), gamma_c=gamma_c) for ny in nys]
    rows = [ref.analytic_rows(ny, p) for ny, p in zip(nys, ps)]
    assert all(np.all(np.isfinite(f)) for r in rows for f in r)
    with lbnlm.Channels(4, nys, ps, "f64", stream=stream) as a, lbnlm.Channels(4, nys, ps, "f64", stream=stream) as b:
        lbnlm.lb_warmstart_apply(a.h)
        warmstart.apply_fields(b, [r[0] for r in rows], [r[2] for r in rows])
        w = np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4)[:, None, None]
        for (na, da), (nb, db) in zip(a.populations(), b.populations()):
            assert np.abs(na - nb).max() <= 1e-13 * np.abs(nb - w).max()
            assert np.abs(da - db).max() <= 1e-13 * max(np.abs(db).max(), 1e-300)
