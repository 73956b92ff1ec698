"""Steps launched back to back (each set up while the one before it still runs) against the same steps with the
device idle between any two: populations, delta rho and monitor bitwise, in the row march, the tile kernel and
pressure-driven ends, on both sides of the size from which a step is launched after the one before."""
import numpy as np
import pytest

from paper_1310_7450_gb300 import inputs, lbnlm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,prec,flags,kw", [
    (1024, 512, "f32", 0, {}), (1000, 777, "bf16", 0, {}), (2048, 2048, "f32", 0, {}), (2048, 2049, "f32", 0, {}),
    (1024, 2049, "bf16", 0, {}), (640, 640, "f32", lbnlm.LB_GRID_TILE_ONLY, {}), (256, 257, "f64", 0, {}),
    (1000, 512, "f32", 0, dict(x_mode="gpbc")), (100, 60, "f32", 0, dict(x_mode="gpbc"))])
def test_back_to_back_steps_equal_separate_ones(nx, ny, prec, flags, kw):
    import torch
    p = dict(inputs.matched_params(0.9, 100.0, 0.1, 1e-3, 1e-5), rho_pert_amp=1e-2, seed=nx + ny)
    out = []
    for apart in (False, True):
        with lbnlm.Channels(nx, ny, p, prec, flags=flags | lbnlm.LB_GRID_NO_GRAPH,
                            stream=torch.cuda.current_stream().cuda_stream, **kw) as sim:
            for _ in range(20):
                sim.step(2)
                if apart:
                    torch.cuda.synchronize()
            out.append(list(sim.populations()[0]) + [sim.monitor()])
            assert list(sim.status()) == [0]
    for x, y in zip(*out):
        assert np.array_equal(x, y)
