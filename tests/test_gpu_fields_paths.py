"""lb_get_fields: every way out gives the same numbers -- host and device buffers, both types, one field at a
time, device buffers off the 16-byte boundary (staged), and the row-march fields pass against the tile
kernel's, at heights and widths where items, strips and vector stores can go wrong."""
import numpy as np
import pytest

from paper_1310_7450_gb300 import inputs, lbnlm

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def stream():
    import torch
    assert torch.cuda.is_available()
    return torch.cuda.current_stream().cuda_stream


def make(nx, ny, prec, flags, stream, **kw):
    p = dict(inputs.matched_params(0.9, 100.0, 0.1, 1e-3, 1e-6), rho_pert_amp=1e-3, seed=4)
    sim = lbnlm.Channels(nx, ny, p, prec, flags=flags, stream=stream, **kw)
    if flags & lbnlm.LB_GRID_RELAXATION_MODEL:
        lbnlm.lb_set_relaxation_model(sim.h, -1, 2.0, 1.0, 50.0)
    if kw.get("walls") == "couette":
        lbnlm.lb_set_wall_velocity(sim.h, -1, 0.01)
    sim.step(7)
    return sim


RX, GN = lbnlm.LB_GRID_RELAXATION_MODEL, lbnlm.LB_GRID_GENERALIZED_NEWTONIAN
CASES = [(128, 16, 0, {}), (128, 17, 0, {}), (384, 131, 0, {}), (256, 48, 0, dict(stress_mode=1)),
         (256, 33, 0, dict(x_mode="gpbc")), (256, 33, 0, dict(walls="couette", stress_mode=1)), (256, 40, GN, {}),
         (256, 40, RX, {}), (256, 40, RX, dict(stress_mode=1))]


@pytest.mark.parametrize("prec", ["f32", "bf16"])
@pytest.mark.parametrize("nx,ny,flags,kw", CASES)
def test_row_march_fields_equal_tile_fields(stream, prec, nx, ny, flags, kw):
    res = []
    for tile in (0, lbnlm.LB_GRID_TILE_ONLY):
        with make(nx, ny, prec, flags | tile, stream, **kw) as sim:
            assert bool(lbnlm.lb_uses_row_march(sim.h)) == (tile == 0)
            before = sim.populations()[0]
            res.append(sim.fields()[0])
            after = sim.populations()[0]
            assert all(np.array_equal(a, b) for a, b in zip(before, after))   # the state is not changed
    for a, b in zip(*res):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("prec,nx,ny", [("f64", 5, [7, 9]), ("f32", 5, [7, 9]), ("f32", 256, 33), ("bf16", 256, 33)])
def test_every_destination_gives_the_same_fields(stream, prec, nx, ny):
    import torch
    with make(nx, ny, prec, 0, stream) as sim:
        n = sim.nodes
        host = [np.zeros(k * n) for k in (2, 4, 1)]
        lbnlm.lb_get_fields(sim.h, *host, 0, False)
        for code, dt, ndt in ((0, torch.float64, np.float64), (1, torch.float32, np.float32)):
            want = [h.astype(ndt) for h in host]
            hst = [np.zeros(k * n, dtype=ndt) for k in (2, 4, 1)]
            lbnlm.lb_get_fields(sim.h, *hst, code, False)
            assert all(np.array_equal(a, b) for a, b in zip(hst, want))
            for off in (0, 1):                     # 1: no 16-byte boundary
                dev = [torch.full((k * n + 1,), 7.0, dtype=dt, device="cuda")[off:off + k * n] for k in (2, 4, 1)]
                lbnlm.lb_get_fields(sim.h, *dev, code, True)
                assert all(np.array_equal(d.cpu().numpy(), b) for d, b in zip(dev, want))
            for k in range(3):                     # one field alone
                one = [None, None, None]
                one[k] = torch.zeros(want[k].size, dtype=dt, device="cuda")
                lbnlm.lb_get_fields(sim.h, *one, code, True)
                assert np.array_equal(one[k].cpu().numpy(), want[k])
