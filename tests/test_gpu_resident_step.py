"""Resident stepping (a small single channel kept on chip for a run of steps) against one launch per step:
populations, delta rho, stress, monitor and fields bitwise, at heights that split unevenly over the
cluster's CTAs, the fewest rows and columns, call lengths around its limits, both stress modes, the moving
wall and a force changed between calls; an unstable channel stops and is reported."""
import numpy as np
import pytest

from paper_1310_7450_gb300 import inputs, lbnlm

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def stream():
    import torch
    assert torch.cuda.is_available()
    return torch.cuda.current_stream().cuda_stream


def run(nx, ny, prec, flags, stream, calls, **kw):
    p = dict(inputs.matched_params(0.9, 50.0, 0.1, 1e-3, 1e-5), rho_pert_amp=1e-3, seed=nx * ny)
    out = []
    with lbnlm.Channels(nx, ny, p, prec, flags=flags | lbnlm.LB_GRID_STORE_SIGMA, stream=stream, **kw) as sim:
        if kw.get("walls") == "couette":
            lbnlm.lb_set_wall_velocity(sim.h, -1, 0.01)
        for k, n in enumerate(calls):
            sim.step(n)
            if n >= 2:
                out.append(sim.monitor())
            lbnlm.lb_set_body_force(sim.h, -1, 1e-5 * (k % 2))
        sig3 = np.zeros(3 * sim.nodes)
        n, d = np.zeros(9 * sim.nodes), np.zeros(sim.nodes)
        lbnlm.lb_get_populations(sim.h, n, d, sig3)
        assert lbnlm.lb_step_count(sim.h) == sum(calls) and list(sim.status()) == [0]
        return out + [n, d, sig3] + list(sim.fields()[0])


@pytest.mark.parametrize("prec", ["f64", "f32", "bf16"])
@pytest.mark.parametrize("nx,ny,kw", [(4, 64, {}), (4, 67, dict(stress_mode=1)), (1, 3, {}), (1, 5, dict(walls="couette")),
                                      (3, 31, {}), (5, 32, dict(walls="couette", stress_mode=1)), (2, 480, {}),
                                      (20, 401, {}), (40, 201, {}), (64, 33, {}), (130, 17, {})])
def test_resident_steps_equal_separate_launches(stream, prec, nx, ny, kw):
    calls = (7, 8, 9, 1, 60, 33, 2)
    a = run(nx, ny, prec, 0, stream, calls, **kw)
    b = run(nx, ny, prec, lbnlm.LB_GRID_NO_GRAPH, stream, calls, **kw)
    for x, y in zip(a, b):
        assert np.array_equal(x, y)


@pytest.mark.parametrize("prec", ["f64", "f32"])
def test_unstable_channel_stops(stream, prec):
    p = dict(inputs.matched_params(0.9, 10.0, 0.1, 1e-3, 3e-3), rho_pert_amp=0.0)   # |u| passes 0.3 after ~100 steps
    with lbnlm.Channels(4, 64, p, prec, stream=stream) as sim:
        sim.step(2000)
        assert list(sim.status()) == [1]
        n, d = sim.populations()[0]
        assert np.all(np.isfinite(n)) and np.all(np.isfinite(d))   # stopped where the guard failed
        assert sim.step(50) == lbnlm.LB_EUNSTABLE
        n2, _ = sim.populations()[0]
        assert np.array_equal(n, n2)
