"""The tensor-core weight gradient at the edges of its tiles: columns of 128 voxels that the
batch does not fill, strips that do not divide H, boxes of one row or plane, every pairing of
channel blocks (16, 32, 64) and channel counts of several blocks, rows with a short last group, and the
general kernel (W < 3). Operands are small integers, so every sum is exact in FP32 in any
order and the comparison has no tolerance."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,D,H,W,K,N", [
    (1, 1, 1, 8, 16, 16), (1, 2, 3, 8, 16, 32), (2, 3, 5, 16, 16, 64), (1, 3, 2, 24, 32, 16), (2, 2, 4, 8, 32, 32),
    (1, 3, 7, 40, 32, 64), (1, 2, 1, 136, 64, 16), (1, 5, 17, 64, 64, 32), (3, 8, 8, 8, 64, 64), (1, 4, 33, 128, 96, 64),
    (1, 6, 19, 32, 64, 96), (1, 2, 9, 72, 128, 96), (2, 24, 40, 40, 32, 32), (1, 1, 2, 256, 128, 128),
    (1, 3, 5, 12, 32, 32), (1, 2, 3, 16, 48, 272), (2, 5, 6, 1, 32, 32), (1, 4, 5, 2, 16, 32), (2, 3, 7, 3, 32, 64),
    (1, 5, 4, 7, 64, 32), (1, 3, 9, 9, 96, 64), (2, 4, 11, 31, 128, 96), (1, 2, 5, 127, 16, 16)])
def test_wgrad_exact_on_integers(B, D, H, W, K, N):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1303_2470_gb300 import mp
    g = torch.Generator(device="cuda")
    g.manual_seed(B + D + H + W + K + N)
    x = torch.randint(-2, 3, (B, D, H, W, K), generator=g, device="cuda").float()
    dy = torch.randint(-2, 3, (B * D * H * W, N), generator=g, device="cuda").float()
    gw = torch.ones((27, K, N), device="cuda")  # the call adds to what is there
    gb = torch.ones(N, device="cuda")
    mp.sg_conv3d_wgrad(x.bfloat16().contiguous(), dy.bfloat16().contiguous(), gw, gb, B, D, H, W, K, N)
    mp.sg_check()
    for t in range(27):
        o = [t // 9 - 1, t // 3 % 3 - 1, t % 3 - 1]
        ref = torch.roll(x, [-v for v in o], (1, 2, 3)).reshape(-1, K).double().T @ dy.double()
        assert torch.equal(gw[t].double(), ref + 1), f"tap {t}"
    assert torch.equal(gb.double(), dy.double().sum(0) + 1)
