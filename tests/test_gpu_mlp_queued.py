"""Training steps and forward passes queued without a host wait (each kernel set up, and part of its operands read,
while the ones before it run) against the same calls with the device idle between any two: predictions,
gradients and parameters bitwise."""
import numpy as np
import pytest

from paper_1310_7450_gb300 import lbnlm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_in,H,n_out,B", [(4, 256, 768, 256), (4, 256, 768, 24), (16, 64, 48, 33), (3, 1000, 70, 512), (1, 1, 1, 1)])
def test_queued_calls_equal_separate_ones(n_in, H, n_out, B):
    import torch
    g = torch.Generator().manual_seed(n_in + H + B)
    x = [torch.randn(B, n_in, generator=g).cuda() for _ in range(3)]
    t = [0.3 * torch.randn(B, n_out, generator=g).cuda() for _ in range(3)]
    out = []
    for apart in (False, True):
        m = lbnlm.lb_mlp_create(n_in, H, n_out, B, 7, torch.cuda.current_stream().cuda_stream)
        wait = torch.cuda.synchronize if apart else (lambda: None)
        try:
            y = [torch.zeros(B, n_out, device="cuda") for _ in range(12)]
            torch.cuda.synchronize()
            for k in range(12):
                lbnlm.lb_mlp_train_step(m, x[k % 3], t[k % 3], B, 1e-2, want_loss=False)
                wait()
                if k % 2:
                    lbnlm.lb_mlp_train_step(m, x[(k + 1) % 3], t[(k + 1) % 3], max(1, B // 2), 1e-2, want_loss=False)
                    wait()
                lbnlm.lb_mlp_forward(m, x[k % 3], B, y[k])
                wait()
            p = np.zeros(lbnlm.lb_mlp_num_params(m), dtype=np.float32)
            lbnlm.lb_mlp_get_params(m, p)
            grad = torch.zeros(p.size, device="cuda")
            loss = lbnlm.lb_mlp_gradients(m, x[0], t[0], B, grad)
            out.append([v.cpu().numpy() for v in y] + [p, grad.cpu().numpy(), np.array(loss)])
        finally:
            lbnlm.lb_mlp_destroy(m)
    for a, b in zip(*out):
        assert np.all(np.isfinite(a)) and np.array_equal(a, b)
