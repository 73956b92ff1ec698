"""A captured lb_get_fields whose buffers go through the handle's staging (addresses that are no multiple of 16), replayed
after calls of the other type have asked for staging of their own: the replay writes the current fields."""
import numpy as np
import pytest

from paper_1310_7450_gb300 import inputs, lbnlm
from stream_capture import Captured

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,prec", [(20, 60, "f32"), (256, 64, "f32"), (33, 40, "f64")])
@pytest.mark.parametrize("captured,other", [(1, 0), (0, 1)])
def test_replay_after_the_other_type(nx, ny, prec, captured, other):
    import torch
    s = torch.cuda.Stream()
    dtype = [torch.float64, torch.float32]
    p = dict(inputs.matched_params(0.9, 50.0, 0.1, 1e-3, 1e-5), rho_pert_amp=1e-3, seed=nx)
    N = nx * ny
    with lbnlm.Channels(nx, ny, p, prec, stream=s.cuda_stream) as sim:
        buf = torch.zeros(7 * N + 1, dtype=dtype[captured], device="cuda")
        out = [buf[1:1 + 2 * N], buf[1 + 2 * N:1 + 6 * N], buf[1 + 6 * N:]]     # (off a 16-byte boundary)
        torch.cuda.synchronize()
        lbnlm.lb_get_fields(sim.h, *out, captured, True)                        # (staging is allocated outside captures)
        torch.cuda.synchronize()
        c = Captured(s.cuda_stream, lambda: lbnlm.lb_get_fields(sim.h, *out, captured, True))
        assert c.status == 0
        for _ in range(3):
            sim.step(2)                                                         # (an even count: the same buffer)
            host = [np.zeros(k * N, dtype=[np.float64, np.float32][other]) for k in (2, 4, 1)]
            lbnlm.lb_get_fields(sim.h, *host, other, False)
            buf.zero_()
            torch.cuda.synchronize()
            c.replay()
            torch.cuda.synchronize()
            for got, want in zip(out, host):
                g = got.cpu().numpy()
                assert np.abs(want).max() > 0 or want.size == 4 * N
                assert np.array_equal(g.astype(np.float32), want.astype(np.float32))
        c.close()
