"""The tensor-core convolutions at the edges of the marching kernel's tiles: a column of 128
voxels that the box does not fill, strips of rows that do not divide H, one-row boxes whose
neighbours are the row itself, several channel blocks, both signs, every compiled channel
count, rows with a short last group, and the general kernel (W < 3). Operands are small integers,
so every sum is exact in FP32 and the comparison has no tolerance; BF16 outputs are the
exact sums rounded once."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,D,H,W,K,N", [
    (1, 1, 1, 8, 16, 16), (1, 2, 3, 8, 16, 32), (2, 3, 5, 16, 32, 32), (1, 3, 2, 24, 96, 48), (2, 2, 4, 8, 64, 32),
    (1, 3, 7, 40, 128, 32), (1, 2, 1, 136, 16, 16), (1, 5, 17, 64, 64, 64), (3, 8, 8, 8, 128, 128),
    (1, 4, 33, 128, 32, 64), (1, 6, 19, 32, 96, 96), (1, 2, 9, 72, 64, 96), (2, 40, 40, 40, 32, 16),
    (1, 1, 2, 256, 128, 96), (1, 3, 4, 16, 48, 32), (1, 3, 5, 12, 32, 32), (1, 2, 3, 16, 64, 272),
    (2, 5, 6, 1, 32, 32), (1, 4, 5, 2, 16, 32), (2, 3, 7, 3, 32, 64), (1, 5, 4, 7, 64, 32), (1, 3, 9, 9, 96, 64),
    (2, 4, 11, 31, 128, 96), (1, 2, 5, 127, 64, 64)])
def test_conv_exact_on_integers(B, D, H, W, K, N):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1303_2470_gb300 import mp
    g = torch.Generator(device="cuda")
    g.manual_seed(B + D + H + W + K + N)
    x = torch.randint(-2, 3, (B, D, H, W, K), generator=g, device="cuda").float()
    w = torch.randint(-2, 3, (27, N, K), generator=g, device="cuda").float()
    bias = torch.randint(-9, 10, (N,), generator=g, device="cuda").float()
    for sign in (1, -1):
        ref = torch.zeros((B, D, H, W, N), dtype=torch.float64, device="cuda")
        for t in range(27):
            o = [sign * (t // 9 - 1), sign * (t // 3 % 3 - 1), sign * (t % 3 - 1)]
            ref += (torch.roll(x, [-v for v in o], (1, 2, 3)).double() @ w[t].double().T)
        ref = (ref + bias).float().reshape(B, -1, N)
        xb, wb = x.bfloat16().reshape(B, -1, K).contiguous(), w.bfloat16().contiguous()
        y = torch.full((B, D * H * W, N), float("nan"), dtype=torch.bfloat16, device="cuda")
        yf = torch.full((B, D * H * W, N), float("nan"), device="cuda")
        mp.sg_conv3d(xb, wb, bias, y, yf, B, D, H, W, K, N, sign, False)
        mp.sg_check()
        assert torch.equal(yf, ref)
        assert torch.equal(y, ref.bfloat16())
        mp.sg_conv3d(xb, wb, bias, y, None, B, D, H, W, K, N, sign, True)
        mp.sg_check()
        assert torch.equal(y, ref.relu().bfloat16())
