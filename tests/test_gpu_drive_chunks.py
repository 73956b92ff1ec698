"""A drive set after create against one given at create, on both sides of the number of channels that one launch
takes, and the monitor's way out to every kind of memory, also from an address that is no multiple of 8."""
import numpy as np
import pytest

from paper_1310_7450_gb300 import inputs, lbnlm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["f32", "f64"])
@pytest.mark.parametrize("n_ch", [1, 31, 127, 128, 129, 300])
def test_drive_set_later_equals_drive_at_create(n_ch, prec):
    import torch
    stream = torch.cuda.current_stream().cuda_stream
    base = dict(inputs.matched_params(0.9, 50.0, 0.1, 1e-3, 1e-5), rho_pert_amp=1e-3, seed=3)
    g = [1e-6 * (c + 1) / n_ch for c in range(n_ch)]
    uw = [1e-2 * (c + 1) / n_ch for c in range(n_ch)]
    out = []
    for later in (True, False):
        ps = [dict(base, g_x=0.0 if later else g[c]) for c in range(n_ch)]
        with lbnlm.Channels(4, [9] * n_ch, ps, prec, walls="couette", stream=stream) as sim:
            for c in range(n_ch):
                lbnlm.lb_set_wall_velocity(sim.h, c, uw[c])
                if later:
                    lbnlm.lb_set_body_force(sim.h, c, g[c])
            sim.step(5)
            mon = sim.monitor()
            dev = torch.zeros(4 * n_ch, dtype=torch.float64, device="cuda")
            pin = torch.zeros(4 * n_ch, dtype=torch.float64).pin_memory()
            raw = torch.zeros(32 * n_ch + 8, dtype=torch.uint8, device="cuda")
            host = np.zeros(4 * n_ch)
            for dst in (dev, pin, raw[4:], host):
                lbnlm.lb_monitor_async(sim.h, dst)
            torch.cuda.synchronize()
            odd = np.frombuffer(raw.cpu().numpy()[4:4 + 32 * n_ch].tobytes(), dtype=np.float64)
            for m in (dev.cpu().numpy(), pin.numpy(), odd, host):
                assert np.array_equal(m.reshape(-1), np.asarray(mon).reshape(-1))
            out.append([np.concatenate([x.reshape(-1) for x in p]) for p in sim.populations()] + [np.asarray(mon)])
    for x, y in zip(*out):
        assert np.array_equal(x, y)
