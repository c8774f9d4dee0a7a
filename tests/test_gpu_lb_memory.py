"""lb_steady where the device has room for everything but its row table (16 bytes a fluid node beside
172): the same flow bit for bit as with room for it. The rest of the device is held by one
allocation for the length of the call."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_flow_without_room_for_the_row_table():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1303_2470_gb300 import mp
    shape = (2048, 150, 150)  # a plane's fluid nodes are within the table's reach
    solid = torch.zeros(shape, dtype=torch.uint8, device="cuda")
    solid[:, :3] = 1  # walls
    nf = solid.numel() - int(solid.sum())
    u, rho = torch.zeros((2, 3) + shape, device="cuda"), torch.zeros((2,) + shape, device="cuda")

    def solve(k):
        with pytest.raises(mp.MPError) as e:
            mp.lb_steady(solid, (1e-5, 0.0, 0.0), u[k], tol=0.0, max_steps=12, check_every=6, rho_out=rho[k],
                         raise_on_unconverged=True)
        assert e.value.code == mp.MP_ENOTCONVERGED

    solve(0)
    mp.mp_release_cached()
    torch.cuda.empty_cache()
    torch.cuda.synchronize()
    # 172 bytes a node, the masks, and what the allocator rounds up or leaves between freed blocks; the
    # table's 16 bytes a node do not fit into what is left then
    room = int(172 * 1.04 * nf) + (150 << 20)
    free = torch.cuda.mem_get_info()[0]
    if free < room + (16 << 20):
        pytest.skip("another program holds the device's memory")
    rest = torch.empty(free - room, dtype=torch.uint8, device="cuda")
    try:
        solve(1)
    finally:
        del rest
        torch.cuda.empty_cache()
        mp.mp_release_cached()
    assert torch.equal(u[0], u[1]) and torch.equal(rho[0], rho[1])
