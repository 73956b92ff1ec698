"""The perceptron's product kernels at the edges of their tiles: batches, widths and depths that are no
multiples of a tile or of a 16-byte piece, a first layer that is evaluated inside the second (few inputs)
and one that is not, depths of several operand slabs, one-element layers.  Against the FP64 reference
with the same BF16 weights, to the bounds of the other perceptron tests; a training step's update
against Adam's formula on the gradients the library reports."""
import numpy as np
import pytest

from oracle import mlp as ref
from paper_1310_7450_gb300 import lbnlm

pytestmark = pytest.mark.gpu

SHAPES = [(1, 1, 1, 1), (4, 256, 768, 24), (16, 40, 33, 31), (17, 40, 36, 33), (3, 260, 1500, 100), (4, 1000, 70, 65),
          (40, 128, 128, 512)]


@pytest.mark.parametrize("n_in,H,n_out,B", SHAPES)
def test_shapes_match_fp64_reference(n_in, H, n_out, B):
    import torch
    rng = np.random.default_rng(n_in + H + B)
    m = lbnlm.lb_mlp_create(n_in, H, n_out, B + 3, 5, torch.cuda.current_stream().cuda_stream)
    try:
        p = np.zeros(lbnlm.lb_mlp_num_params(m), dtype=np.float32)
        lbnlm.lb_mlp_get_params(m, p)
        p += rng.normal(0, 0.02, p.size).astype(np.float32)   # (biases too)
        lbnlm.lb_mlp_set_params(m, p)
        x = rng.normal(0, 1, (B, n_in)).astype(np.float32)
        t = rng.normal(0, 0.3, (B, n_out)).astype(np.float32)
        xd, td = torch.tensor(x, device="cuda"), torch.tensor(t, device="cuda")
        buf = torch.zeros(B * n_out + 1, device="cuda")
        y = buf[1:]                                            # (4-byte aligned only)
        lbnlm.lb_mlp_forward(m, xd, B, y)
        g = torch.zeros(p.size, device="cuda")
        loss = lbnlm.lb_mlp_gradients(m, xd, td, B, g)
        y_ref, _ = ref.forward(p, x, n_in, H, n_out, bf16=True)
        loss_ref, g_ref = ref.loss_and_grad(p, x, t, n_in, H, n_out, bf16=True)
        assert np.abs(y.cpu().numpy().reshape(B, n_out) - y_ref).max() <= 1e-5 * max(1.0, np.abs(y_ref).max())
        assert loss == pytest.approx(loss_ref, rel=1e-5)
        gg = g.cpu().numpy()
        assert np.abs(gg - g_ref).max() <= 1e-4 * np.abs(g_ref).max()
        # first Adam step: m/c1 = g, v/c2 = g^2
        lr = 1e-3
        assert lbnlm.lb_mlp_train_step(m, xd, td, B, lr) == pytest.approx(loss_ref, rel=1e-5)
        q = np.zeros_like(p)
        lbnlm.lb_mlp_get_params(m, q)
        want = p.astype(np.float64) - lr * gg.astype(np.float64) / (np.abs(gg.astype(np.float64)) + 1e-8)
        big = np.abs(gg) > 1e-6 * np.abs(gg).max()             # (the sign of a rounded zero is open)
        assert np.abs(q - want)[big].max() <= 1e-3 * lr + 1e-7
        y2 = torch.zeros(B, n_out, device="cuda")
        lbnlm.lb_mlp_forward(m, xd, B, y2)                     # the BF16 copies followed
        y_ref, _ = ref.forward(q, x, n_in, H, n_out, bf16=True)
        assert np.abs(y2.cpu().numpy() - y_ref).max() <= 1e-5 * max(1.0, np.abs(y_ref).max())
    finally:
        lbnlm.lb_mlp_destroy(m)
