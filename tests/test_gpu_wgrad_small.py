"""The weight gradient at the sizes where it passes from the general kernel to the tensor-core one: 128
voxels, 256 with blocks of 64 input channels. Integers: exact in any order."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,D,H,W", [(1, 1, 42, 3), (2, 4, 4, 4), (1, 1, 43, 3), (1, 3, 17, 5), (2, 2, 8, 8), (1, 1, 37, 7)])
@pytest.mark.parametrize("K,N", [(16, 32), (64, 32), (64, 64), (96, 48)])
def test_wgrad_exact_on_small_boxes(B, D, H, W, K, N):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1303_2470_gb300 import mp
    g = torch.Generator(device="cuda")
    g.manual_seed(B + D + H + W + K + N)
    x = torch.randint(-2, 3, (B, D, H, W, K), generator=g, device="cuda").float()
    dy = torch.randint(-2, 3, (B * D * H * W, N), generator=g, device="cuda").float()
    gw, gb = torch.zeros((27, K, N), device="cuda"), torch.zeros(N, device="cuda")
    mp.sg_conv3d_wgrad(x.bfloat16().contiguous(), dy.bfloat16().contiguous(), gw, gb, B, D, H, W, K, N)
    mp.sg_check()
    for t in range(27):
        o = [t // 9 - 1, t // 3 % 3 - 1, t % 3 - 1]
        ref = torch.roll(x, [-v for v in o], (1, 2, 3)).reshape(-1, K).double().T @ dy.double()
        assert torch.equal(gw[t].double(), ref), f"tap {t}"
    assert torch.equal(gb.double(), dy.double().sum(0))
