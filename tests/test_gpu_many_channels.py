"""Drive of handles with more channels than one block has threads: a force (wall velocity) given to all channels and
then to single ones, at the edges of the blocks, against the same values given at create."""
import numpy as np
import pytest

from paper_1310_7450_gb300 import inputs, lbnlm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,kw", [("f32", {}), ("f64", dict(walls="couette")), ("f32", dict(x_mode="gpbc"))])
def test_all_then_single_channels(prec, kw):
    import torch
    stream = torch.cuda.current_stream().cuda_stream
    n_ch, base = 1500, dict(inputs.matched_params(0.9, 50.0, 0.1, 1e-3, 0.0), rho_pert_amp=1e-3, seed=3)
    g, uw = np.full(n_ch, 2e-6), np.full(n_ch, 1e-2)
    single = [0, 1, 127, 128, 129, 1023, 1024, 1499]
    for k, c in enumerate(single):
        g[c], uw[c] = 1e-6 * (k + 3), 1e-3 * (k + 1)
    out = []
    for later in (True, False):
        ps = [dict(base, g_x=0.0 if later else g[c]) for c in range(n_ch)]
        if later and kw.get("x_mode") == "gpbc":
            start = [dict(base, g_x=g[c]) for c in range(n_ch)]       # (the force also sets the starting density)
            with lbnlm.Channels(4, [5] * n_ch, start, prec, stream=stream, **kw) as ref:
                pops = ref.populations()
        with lbnlm.Channels(4, [5] * n_ch, ps, prec, stream=stream, **kw) as sim:
            if later:
                lbnlm.lb_set_body_force(sim.h, -1, 2e-6)
                for c in single:
                    lbnlm.lb_set_body_force(sim.h, c, g[c])
                if kw.get("x_mode") == "gpbc":
                    sim.set_populations([p[0] for p in pops], [p[1] for p in pops])
            elif kw.get("x_mode") == "gpbc":
                pops = sim.populations()
                sim.set_populations([p[0] for p in pops], [p[1] for p in pops])
            if kw.get("walls") == "couette":
                for c in range(n_ch) if not later else []:
                    lbnlm.lb_set_wall_velocity(sim.h, c, uw[c])
                if later:
                    lbnlm.lb_set_wall_velocity(sim.h, -1, 1e-2)
                    for c in single:
                        lbnlm.lb_set_wall_velocity(sim.h, c, uw[c])
            sim.step(5)
            out.append([np.concatenate([x.reshape(-1) for x in p]) for p in sim.populations()] + [sim.monitor()])
    for x, y in zip(*out):
        assert np.array_equal(x, y)
