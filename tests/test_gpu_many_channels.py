"""Handles with more channels than one block has threads.  Their drive: a force (wall velocity) given to all channels and
then to single ones, at the edges of the blocks, against the same values given at create.  Their monitor, into
device and pinned memory, against the blocking call."""
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


@pytest.mark.parametrize("n_ch", [31, 32, 33, 1500])
def test_monitor_reaches_every_kind_of_memory(n_ch):
    import torch
    p = dict(inputs.matched_params(0.9, 50.0, 0.1, 1e-3, 1e-5), rho_pert_amp=1e-3)
    with lbnlm.Channels(4, [5] * n_ch, [dict(p, seed=c + 1) for c in range(n_ch)], "f32",
                        stream=torch.cuda.current_stream().cuda_stream) as sim:
        sim.step(4)
        want = np.asarray(sim.monitor()).reshape(-1)
        assert len(set(want[1::4])) > n_ch // 2                            # (channels differ)
        dev = torch.zeros(4 * n_ch + 2, dtype=torch.float64, device="cuda")
        pin = torch.zeros(4 * n_ch + 2, dtype=torch.float64).pin_memory()
        for dst in (dev, pin):
            lbnlm.lb_monitor_async(sim.h, dst[1:-1])
        torch.cuda.synchronize()
        for got in (dev.cpu().numpy(), pin.numpy()):
            assert np.array_equal(got[1:-1], want) and got[0] == got[-1] == 0.0
