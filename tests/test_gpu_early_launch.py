"""Single steps launched back to back, each set up while the one before it runs, against the same steps with the
device idle before each of them: populations, delta rho, fields and monitor bitwise, in the tile kernel and the
row march of each precision.  (LB_MONITOR_FLUX_MAX gives one-step calls a monitor.)"""
import numpy as np
import pytest

from paper_1310_7450_gb300 import inputs, lbnlm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,prec,flags,kw", [
    (1024, 512, "f32", 0, {}), (1000, 777, "bf16", 0, {}), (1001, 777, "f32", 0, dict(stress_mode=1)),
    (640, 640, "f32", lbnlm.LB_GRID_TILE_ONLY, {}), (640, 640, "bf16", lbnlm.LB_GRID_TILE_ONLY, {}),
    (1000, 512, "bf16", 0, dict(x_mode="gpbc")), (256, 2048, "bf16", 0, dict(x_mode="gpbc", stress_mode=1)),
    (100, 300, "f32", 0, dict(walls="couette", stress_mode=1)), (256, 257, "f64", 0, {}), (100, 60, "f32", 0, dict(x_mode="gpbc")),
    (256, 200, "bf16", lbnlm.LB_GRID_STRESS_DIVERGENCE, {}), (1024, 300, "f32", lbnlm.LB_GRID_RELAXATION_MODEL, {})])
def test_steps_launched_early_equal_steps_alone(nx, ny, prec, flags, kw):
    import torch
    p = dict(inputs.matched_params(0.9, 100.0, 0.1, 1e-3, 1e-5), rho_pert_amp=1e-2, seed=nx + ny)
    out = []
    for alone in (False, True):
        with lbnlm.Channels(nx, ny, p, prec, flags=flags | lbnlm.LB_GRID_NO_GRAPH,
                            stream=torch.cuda.current_stream().cuda_stream, **kw) as sim:
            lbnlm.lb_set_monitor_mode(sim.h, lbnlm.LB_MONITOR_FLUX_MAX)
            if flags & lbnlm.LB_GRID_RELAXATION_MODEL:
                lbnlm.lb_set_relaxation_model(sim.h, -1, 2.0, 1.0, 50.0)
            torch.cuda.synchronize()
            if alone:
                for _ in range(40):
                    sim.step(1)
                    torch.cuda.synchronize()
            else:
                sim.step(40)
            out.append(list(sim.populations()[0]) + list(sim.fields()[0]) + [sim.monitor()])
            assert list(sim.status()) == [0]
    for x, y in zip(*out):
        assert np.array_equal(x, y)
