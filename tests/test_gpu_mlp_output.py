"""lb_mlp_forward into every place that a copy reached before the last layer wrote its results itself: device addresses
that are multiples of nothing, and the network's input.  Bitwise the same values as into memory of its own."""
import pytest

from paper_1310_7450_gb300 import lbnlm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("offset", [1, 2, 3, 4, 6])
@pytest.mark.parametrize("B", [1, 33])
def test_any_address(offset, B):
    import torch
    m = lbnlm.lb_mlp_create(4, 40, 24, 40, 3, torch.cuda.current_stream().cuda_stream)
    try:
        x = torch.randn(B, 4, generator=torch.Generator().manual_seed(B)).cuda()
        want = torch.zeros(B, 24, device="cuda")
        lbnlm.lb_mlp_forward(m, x, B, want)
        raw = torch.zeros(4 * B * 24 + 16, dtype=torch.uint8, device="cuda")
        lbnlm.lb_mlp_forward(m, x, B, raw[offset:])
        torch.cuda.synchronize()
        got = raw[offset:offset + 4 * B * 24].clone().view(torch.float32).reshape(B, 24)
        assert torch.equal(got, want) and want.abs().max() > 0
        assert not raw[:offset].any() and not raw[offset + 4 * B * 24:].any()
    finally:
        lbnlm.lb_mlp_destroy(m)


@pytest.mark.parametrize("n,B", [(8, 50), (24, 7)])
def test_output_over_the_input(n, B):
    import torch
    m = lbnlm.lb_mlp_create(n, 48, n, B, 3, torch.cuda.current_stream().cuda_stream)
    try:
        x = torch.randn(B, n, generator=torch.Generator().manual_seed(B)).cuda()
        want = torch.zeros(B, n, device="cuda")
        lbnlm.lb_mlp_forward(m, x, B, want)
        lbnlm.lb_mlp_forward(m, x, B, x)
        assert torch.equal(x, want)
    finally:
        lbnlm.lb_mlp_destroy(m)
