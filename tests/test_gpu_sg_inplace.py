"""sg_pool2_grad_relu with its output in place of its fine input, as the network's backward pass
calls it, against the same call with an output of its own: the same values bit for bit."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,D,H,W,C", [(1, 2, 2, 2, 8), (3, 6, 10, 14, 96), (2, 48, 40, 32, 32), (1, 64, 64, 64, 64)])
def test_masked_pool_gradient_in_place(B, D, H, W, C):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1303_2470_gb300 import mp
    gen = torch.Generator(device="cuda")
    gen.manual_seed(D + C)
    n = B * D * H * W * C
    dy, g, act = (torch.randn(k, generator=gen, device="cuda").bfloat16() for k in (n // 8, n, n))
    out = torch.full_like(g, 9)
    mp.sg_pool2_grad_relu(dy, g, act, out, B, D, H, W, C)
    for _ in range(3):
        inplace = g.clone()
        mp.sg_pool2_grad_relu(dy, inplace, act, inplace, B, D, H, W, C)
        assert torch.equal(inplace, out)
