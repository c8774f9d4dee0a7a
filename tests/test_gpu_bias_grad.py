"""The bias gradient where its blocks sum few voxels (64 and a little more), a last block of one, many
channels and more than one block of channels. Integers: exact in any order."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("V,N", [(1, 16), (64, 256), (65, 272), (4096, 256), (19457, 32), (20001, 48), (311_297, 16),
                                 (400, 2064)])
def test_bias_gradient_exact_on_integers(V, N):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1303_2470_gb300 import mp
    g = torch.Generator(device="cuda")
    g.manual_seed(V + N)
    x = torch.zeros((V, 16), dtype=torch.bfloat16, device="cuda")
    dy = torch.randint(-2, 3, (V, N), generator=g, device="cuda").float()
    gw, gb = torch.zeros((27, 16, N), device="cuda"), torch.ones(N, device="cuda")
    mp.sg_conv3d_wgrad(x, dy.bfloat16(), gw, gb, 1, 1, V, 1, 16, N)
    mp.sg_check()
    assert torch.equal(gb.double(), dy.double().sum(0) + 1) and not gw.any()
