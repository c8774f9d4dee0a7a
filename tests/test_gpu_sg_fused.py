"""The fused forms of the network's passes (upsampled input, skip sum, ReLU mask, masked pool and
upsampling gradients) against the separate calls: the same values bit for bit. Boxes of
widths and channel counts that the marching and the general convolution take, channel counts that the
16-byte passes do and do not take, buffers off a 16-byte boundary, and the loss gradient with
and without its vector form."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
BF = torch.bfloat16


@pytest.fixture(scope="module")
def mp():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1303_2470_gb300 import mp as m
    return m


def _rand(g, *shape):
    return torch.randn(shape, generator=g, device="cuda").to(BF)


@pytest.mark.parametrize("B,D,H,W,K,N", [(1, 2, 4, 8, 16, 32), (2, 4, 6, 16, 64, 32), (2, 4, 2, 12, 32, 16),
                                         (1, 6, 10, 24, 96, 64), (1, 4, 6, 2, 64, 32),
                                         (1, 2, 4, 10, 48, 32)])
def test_fused_convolution_equals_separate_calls(mp, B, D, H, W, K, N):
    g = torch.Generator(device="cuda")
    g.manual_seed(K + N)
    V = D * H * W
    xc, w, bias = _rand(g, B, V // 8, K), _rand(g, 27, N, K), torch.randn(N, generator=g, device="cuda")
    other = _rand(g, B, V, N).relu()
    xu = torch.empty((B, V, K), dtype=BF, device="cuda")
    mp.sg_up2(xc, xu, B, D // 2, H // 2, W // 2, K)
    for sign in (1, -1):
        y = torch.empty((B, V, N), dtype=BF, device="cuda")
        mp.sg_conv3d(xu, w, bias, y, None, B, D, H, W, K, N, sign, True)
        total, masked = torch.empty_like(y), y.clone()
        mp.sg_add(y, other, total, y.numel())
        mp.sg_relu_grad(other, masked, y.numel())
        for mode, ref in ((1, total), (2, masked)):
            for up, x in ((False, xu), (True, xc)):
                y1, y2 = torch.full_like(y, 9), torch.full_like(y, 9)
                mp.sg_conv3d_ex(x, w, bias, y1, None, y2, other, mode, up, B, D, H, W, K, N, sign, True)
                assert torch.equal(y1, y) and torch.equal(y2, ref)
                y2.fill_(9)
                mp.sg_conv3d_ex(x, w, bias, None, None, y2, other, mode, up, B, D, H, W, K, N, sign, True)
                assert torch.equal(y2, ref)
    # integers: the weight gradient is exact in any order
    xi = torch.randint(-2, 3, (B, V // 8, K), generator=g, device="cuda").to(BF)
    dy = torch.randint(-2, 3, (B, V, N), generator=g, device="cuda").to(BF)
    mp.sg_up2(xi, xu, B, D // 2, H // 2, W // 2, K)
    ga, gb = torch.zeros((27, K, N), device="cuda"), torch.zeros((27, K, N), device="cuda")
    mp.sg_conv3d_wgrad(xu, dy, ga, None, B, D, H, W, K, N)
    mp.sg_conv3d_wgrad_ex(xi, dy, gb, None, True, B, D, H, W, K, N)
    assert torch.equal(ga, gb)
    mp.sg_check()
    for bad in (dict(mode=1, y2=None), dict(mode=0, y2=other), dict(mode=3, y2=other)):
        with pytest.raises(mp.MPError) as e:
            mp.sg_conv3d_ex(xu, w, bias, None, None, bad["y2"], other, bad["mode"], False, B, D, H, W, K, N)
        assert e.value.code == mp.MP_EINVAL


@pytest.mark.parametrize("B,D,H,W,C", [(1, 1, 1, 1, 8), (2, 3, 5, 2, 32), (1, 2, 3, 4, 96), (2, 2, 2, 3, 6)])
def test_pooling_passes(mp, B, D, H, W, C):
    """Against plain torch; D, H, W coarse."""
    g = torch.Generator(device="cuda")
    g.manual_seed(C)
    V = D * H * W
    for off in (0, 2):  # off: buffers 4 bytes off a 16-byte boundary take the general kernels
        def buf(n):
            return torch.empty(n + 8, dtype=BF, device="cuda")[off:off + n]
        fine, coarse = buf(B * 8 * V * C), buf(B * V * C)
        fine.copy_(_rand(g, fine.numel()))
        coarse.copy_(_rand(g, coarse.numel()))
        f = fine.view(B, D, 2, H, 2, W, 2, C)
        out_c, out_f = buf(coarse.numel()), buf(fine.numel())
        s = None
        for k in range(8):  # the order of the kernels' FP32 sums
            v = f[:, :, k >> 2, :, (k >> 1) & 1, :, k & 1].float()
            s = v if s is None else s + v
        mp.sg_pool2(fine, out_c, B, 2 * D, 2 * H, 2 * W, C)
        assert torch.equal(out_c, (s * 0.125).to(BF).reshape(-1))
        mp.sg_up2_grad(fine, out_c, B, D, H, W, C)
        assert torch.equal(out_c, s.to(BF).reshape(-1))
        c8 = coarse.view(B, D, 1, H, 1, W, 1, C).expand(B, D, 2, H, 2, W, 2, C)
        mp.sg_up2(coarse, out_f, B, D, H, W, C)
        assert torch.equal(out_f, c8.reshape(-1))
        pg = (c8.float() * 0.125).to(BF).reshape(-1)
        mp.sg_pool2_grad(coarse, out_f, B, 2 * D, 2 * H, 2 * W, C)
        assert torch.equal(out_f, pg)
        t = buf(fine.numel())
        mp.sg_add(fine, pg.contiguous(), t, t.numel())
        assert torch.equal(t, (fine.float() + pg.float()).to(BF))
        if C % 8 or off:
            with pytest.raises(mp.MPError):
                mp.sg_up2_grad_relu(fine, coarse, out_c, B, D, H, W, C)
            continue
        act_c, act_f = _rand(g, coarse.numel()), _rand(g, fine.numel())
        mp.sg_up2_grad_relu(fine, act_c, out_c, B, D, H, W, C)
        assert torch.equal(out_c, torch.where(act_c > 0, s.to(BF).reshape(-1), torch.zeros((), dtype=BF, device="cuda")))
        ref = torch.where(act_f > 0, t, torch.zeros((), dtype=BF, device="cuda"))
        mp.sg_pool2_grad_relu(coarse, fine, act_f, fine, B, 2 * D, 2 * H, 2 * W, C)
        assert torch.equal(fine, ref)


@pytest.mark.parametrize("V,ldy,nc", [(1, 16, 4), (1000, 16, 4), (700_001, 16, 4), (333, 16, 3), (50, 12, 4)])
def test_masked_loss_gradient(mp, V, ldy, nc):
    g = torch.Generator(device="cuda")
    g.manual_seed(V)
    y = torch.randn((1, V, ldy), generator=g, device="cuda")
    t = torch.randn((1, V, nc), generator=g, device="cuda")
    x = torch.zeros((1, V, 16), dtype=BF, device="cuda")
    x[:, :, 0] = (torch.rand((1, V), generator=g, device="cuda") < 0.6).to(BF)
    loss = torch.zeros(1, dtype=torch.float64, device="cuda")
    dy = torch.empty((1, V, ldy), dtype=BF, device="cuda")
    mp.sg_mse(y, ldy, t, nc, x, dy, loss, 1, V, 7.0)
    d = (y[:, :, :nc] - t) * x[:, :, :1].float()
    ref = torch.zeros((1, V, ldy), device="cuda")
    ref[:, :, :nc] = float(torch.tensor(2.0 / (nc * 7.0), dtype=torch.float32)) * d
    assert torch.equal(dy, ref.to(BF))
    want = float((d.double() ** 2).sum()) / (nc * 7.0)
    assert abs(loss.item() - want) <= 1e-12 * want
