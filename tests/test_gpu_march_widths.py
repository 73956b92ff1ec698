"""Row-march kernel at widths that are no whole strips: narrower last strips, rows that are and are not a
multiple of 16 bytes, odd widths, one strip and several, in every variant.  Its populations, delta rho,
fields and monitor against the tile kernel's (the same arithmetic: populations and stress bitwise but
for the relaxation-time extensions; the monitor's FP32 sums to their rounding)."""
import numpy as np
import pytest

from paper_1310_7450_gb300 import inputs, lbnlm

pytestmark = pytest.mark.gpu

RX, GN, SR = lbnlm.LB_GRID_RELAXATION_MODEL, lbnlm.LB_GRID_GENERALIZED_NEWTONIAN, lbnlm.LB_GRID_BF16_STOCHASTIC


@pytest.fixture(scope="module")
def stream():
    import torch
    assert torch.cuda.is_available()
    return torch.cuda.current_stream().cuda_stream


def run(nx, ny, prec, flags, stream, steps=9, **kw):
    p = dict(inputs.matched_params(0.9, 100.0, 0.1, 1e-3, 1e-5), rho_pert_amp=1e-2, seed=nx + ny)
    with lbnlm.Channels(nx, ny, p, prec, flags=flags | lbnlm.LB_GRID_STORE_SIGMA, stream=stream, **kw) as sim:
        if flags & RX:
            lbnlm.lb_set_relaxation_model(sim.h, -1, 2.0, 1.0, 50.0)
        if kw.get("walls") == "couette":
            lbnlm.lb_set_wall_velocity(sim.h, -1, 0.01)
        sim.step(steps)
        mon = sim.monitor()[0]
        lbnlm.lb_set_monitor_mode(sim.h, lbnlm.LB_MONITOR_FLUX_MAX)
        sim.step(1)
        mon2 = sim.monitor()[0]
        march = bool(lbnlm.lb_uses_row_march(sim.h))
        return march, sim.populations()[0], sim.fields()[0], mon, mon2, list(sim.status())


def same(nx, ny, prec, flags, stream, **kw):
    a = run(nx, ny, prec, flags, stream, **kw)
    b = run(nx, ny, prec, flags | lbnlm.LB_GRID_TILE_ONLY, stream, **kw)
    assert a[0] and not b[0]
    for x, y in zip(a[1] + a[2][1:2], b[1] + b[2][1:2]):
        if flags & RX:   # (one product of the force terms rounds differently in about one of 3e7 node updates)
            assert np.abs(x - y).max() <= 2.0 ** -18 * np.abs(y).max() and np.mean(x != y) < 1e-3
        else:
            assert np.array_equal(x, y)
    # u and rho are read out through the hydrodynamic density, one more rounding of a number near 1
    assert np.abs(a[2][2] - b[2][2]).max() <= 2.0 ** -23
    assert np.abs(a[2][0] - b[2][0]).max() <= 2.0 ** -22 * np.abs(b[2][0]).max()
    assert a[5] == b[5] == [0]
    # FP32 sums of at most nx * ny terms in another order
    for x, y in zip(a[3:5], b[3:5]):
        np.testing.assert_allclose(x[[2, 3]], y[[2, 3]], rtol=1e-6)
        assert abs(x[0] - y[0]) <= 1e-5 * abs(y[0])
        assert abs(x[1] - y[1]) <= 1e-5 * ny * y[2]


# rows of 16-byte multiples in both precisions (200, 1000), in FP32 only (196, 132), in neither; last strips of
# few columns (8194: two; 8193 would leave one); whole strips cut into items of two or three rows
WIDTHS = [(200, 2101), (1000, 447), (196, 2133), (132, 3101), (130, 3133), (129, 3141), (255, 1601), (257, 1617),
          (100, 4101), (97, 4153), (385, 1101), (1030, 433), (8193, 53), (8194, 53), (128, 16), (128, 17), (256, 515)]


@pytest.mark.parametrize("prec", ["f32", "bf16"])
@pytest.mark.parametrize("nx,ny", WIDTHS)
def test_widths_equal_tile_kernel(stream, prec, nx, ny):
    same(nx, ny, prec, 0, stream)


@pytest.mark.parametrize("prec", ["f32", "bf16"])
@pytest.mark.parametrize("nx,ny", [(200, 2103), (131, 3103), (97, 4207)])
@pytest.mark.parametrize("flags,kw", [(0, dict(stress_mode=1)), (0, dict(x_mode="gpbc")), (0, dict(walls="couette")),
                                      (0, dict(x_mode="gpbc", walls="couette", stress_mode=1)), (GN, {}), (RX, {}),
                                      (RX, dict(stress_mode=1)), (SR, {})])
def test_variants_equal_tile_kernel(stream, prec, nx, ny, flags, kw):
    if flags == SR and prec != "bf16":
        pytest.skip("stochastic rounding is a BF16 option")
    same(nx, ny, prec, flags, stream, **kw)
