"""The tensor-core weight gradient where a block takes three and more units shorter than its rings
of staged rows (the coarser levels of 48^3 and 64^3 training boxes), a short last strip, and one or two
accumulator sets, with x as it is and read as its upsampling. Small integers: every sum is
exact in FP32 in any order and the comparison has no tolerance."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,D,H,W,K,N", [
    (4, 12, 12, 12, 96, 96), (4, 12, 12, 12, 128, 96), (1, 48, 48, 48, 32, 32), (1, 48, 48, 48, 32, 16),
    (2, 16, 16, 16, 96, 96), (4, 18, 7, 118, 32, 16), (4, 64, 4, 128, 32, 32), (3, 20, 34, 30, 64, 32),
    (2, 24, 18, 40, 64, 64), (1, 40, 33, 64, 16, 16), (4, 32, 6, 64, 64, 32), (4, 24, 9, 80, 64, 32),
    (4, 32, 6, 64, 128, 64)])
def test_wgrad_exact_over_many_units(B, D, H, W, K, N):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1303_2470_gb300 import mp
    g = torch.Generator(device="cuda")
    g.manual_seed(B + D + H + W + K + N)
    dy = torch.randint(-2, 3, (B * D * H * W, N), generator=g, device="cuda").float()
    for up in (False, True):
        if up and (D % 2 or H % 2 or W % 2):
            continue
        s = 2 if up else 1
        stored = torch.randint(-2, 3, (B, D // s, H // s, W // s, K), generator=g, device="cuda").float()
        x = stored
        for axis in (1, 2, 3):
            x = x.repeat_interleave(s, axis)
        gw = torch.zeros((27, K, N), device="cuda")
        mp.sg_conv3d_wgrad_ex(stored.bfloat16().contiguous(), dy.bfloat16().contiguous(), gw, None, up, B, D, H, W, K, N)
        mp.sg_check()
        for t in range(27):
            o = [t // 9 - 1, t // 3 % 3 - 1, t % 3 - 1]
            ref = torch.roll(x, [-v for v in o], (1, 2, 3)).reshape(-1, K).double().T @ dy.double()
            assert torch.equal(gw[t].double(), ref), f"up {up}, tap {t}"
