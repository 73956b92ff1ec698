"""lb_warmstart_apply at the edges of its kernels' ranges: odd and even heights (the profile is evaluated
for one half), fewer and more rows than a block takes at once, widths on both sides of the limit where
the writes change shape; every stress mode's and boundary's start.  Against lb_set_fields with the
reference profiles, to the FP64 bound of the other warm-start tests (1e-13)."""
import numpy as np
import pytest

import warmstart_reference as ref
from paper_1310_7450_gb300 import inputs, lbnlm, warmstart

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def stream():
    import torch
    assert torch.cuda.is_available()
    return torch.cuda.current_stream().cuda_stream


@pytest.mark.parametrize("nx,nys,kw", [(1, [3, 4, 257], {}), (64, [5, 300], {}), (65, [16, 31], {}), (130, [700], {}),
                                       (4, [33, 1024], dict(stress_mode=1)), (6, [48], dict(x_mode="gpbc"))])
@pytest.mark.parametrize("network", [False, True])
def test_start_state_equals_set_fields(stream, nx, nys, kw, network):
    import torch
    ps = [dict(inputs.yield_stress_channel(ny, theta=10.0 * (k + 1), g_x=2e-7 * (64.0 / ny) ** 2)) for k, ny in enumerate(nys)]
    raw = np.random.default_rng(nx).normal(0.0, 0.05, (len(nys), 3 * ref.NPTS)).astype(np.float32)
    with lbnlm.Channels(nx, nys, ps, "f64", stream=stream, **kw) as a, lbnlm.Channels(nx, nys, ps, "f64", stream=stream, **kw) as b:
        a.step(3)   # (a carried stress and a flow-induced density to be overwritten)
        if network:
            lbnlm.lb_warmstart_apply(a.h, torch.tensor(raw, device="cuda"))
            prof = ref.decode(nys, ps, raw.astype(np.float64))
            warmstart.apply_fields(b, [ref.to_rows(f[0], ny) for f, ny in zip(prof, nys)],
                                   [ref.to_rows(f[2], ny) for f, ny in zip(prof, nys)])
        else:
            lbnlm.lb_warmstart_apply(a.h)
            rows = [ref.analytic_rows(ny, p) for ny, p in zip(nys, ps)]
            warmstart.apply_fields(b, [r[0] for r in rows], [r[2] for r in rows])
        w = np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4)[:, None, None]
        for (na, da), (nb, db) in zip(a.populations(), b.populations()):
            assert np.abs(na - nb).max() <= 1e-13 * np.abs(nb - w).max()
            assert np.abs(da - db).max() <= 1e-13 * max(np.abs(db).max(), 1e-300)
        a.step(2)
        b.step(2)
        for (ua, sa, _), (ub, sb, _) in zip(a.fields(), b.fields()):
            assert np.abs(ua - ub).max() <= 1e-12 * np.abs(ub).max()
            assert np.abs(sa - sb).max() <= 1e-11 * np.abs(sb).max()
