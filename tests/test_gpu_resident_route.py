"""Which small channels take runs of steps on chip: those that fit one cluster (lb_step then replays no captured graph in a
60-step call), over the shapes whose results the comparison with separate launches covers, and a wide one that
fits (its results compared here)."""
import numpy as np
import pytest

from paper_1310_7450_gb300 import inputs, lbnlm

pytestmark = pytest.mark.gpu


def stream():
    import torch
    return torch.cuda.current_stream().cuda_stream


def params(nx, ny):
    return dict(inputs.matched_params(0.9, 50.0, 0.1, 1e-3, 1e-5), rho_pert_amp=1e-3, seed=nx * ny)


ALWAYS = [(4, 64, {}), (4, 67, dict(stress_mode=1)), (1, 3, {}), (1, 5, dict(walls="couette")), (3, 31, {}),
          (5, 32, dict(walls="couette", stress_mode=1)), (2, 480, {}), (7, 90, {}), (4, 250, {})]
NOT_F64 = [(20, 401, {}), (40, 201, {}), (64, 33, {}), (160, 32, {})]     # (more than 128 threads per CTA)
NEVER = [(130, 17, {}), (150, 33, {}), (4, 64, dict(x_mode="gpbc"))]


@pytest.mark.parametrize("prec", ["f64", "f32", "bf16"])
def test_shapes_that_stay_on_chip(prec):
    for shapes, resident in ((ALWAYS, True), (NOT_F64, prec != "f64"), (NEVER, False)):
        for nx, ny, kw in shapes:
            with lbnlm.Channels(nx, ny, params(nx, ny), prec, stream=stream(), **kw) as sim:
                sim.step(60)
                assert (lbnlm.lb_graph_replays(sim.h) == 0) == resident, (nx, ny, kw)


@pytest.mark.parametrize("prec", ["f32", "bf16"])
@pytest.mark.parametrize("nx,ny,mode", [(160, 32, 0), (160, 33, 1), (130, 34, 0)])
def test_wide_shapes_equal_separate_launches(prec, nx, ny, mode):
    out = []
    for flags in (0, lbnlm.LB_GRID_NO_GRAPH):
        with lbnlm.Channels(nx, ny, params(nx, ny), prec, flags=flags, stream=stream(), stress_mode=mode) as sim:
            for n in (7, 8, 33, 2):
                sim.step(n)
            out.append(list(sim.populations()[0]) + list(sim.fields()[0]) + [sim.monitor()])
    for a, b in zip(*out):
        assert np.array_equal(a, b)
