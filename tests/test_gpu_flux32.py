"""The flux step of one context stepped on its own against the same context in a group (two
bodies of one update): the same fields bit for bit, Z and D up to the order of FP64 sums of the
same FP32 terms. Node counts at the edges of warps and blocks, one chunk of species, two and
more, padded species, one to three moments; runs split around graph replays, and steps
alternating between the group and the context, which share the series position."""
import numpy as np
import pytest

from paper_1303_2470_gb300 import media

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,directions,species", [
    ((3, 3, 3), "x", 1), ((4, 8, 8), "xz", 1), ((9, 11, 13), "xyz", 1), ((8, 8, 4), "y", 4), ((17, 9, 5), "x", 5),
    ((7, 12, 11), "x", 32), ((8, 6, 11), "xz", 2), ((9, 7, 10), "xyz", 7), ((40, 33, 31), "x", 3)])
def test_own_steps_equal_grouped_steps(shape, directions, species):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1303_2470_gb300 import mp
    solid = media.bulk(*shape[::-1]) if min(shape) < 4 else media.random_spheres(shape, 2, 0.7, seed=41)[0]
    u = torch.as_tensor(media.random_flow(solid, 0.01, seed=42).astype(np.float32)).cuda()
    Db, ka, kd = media.species(species, seed=43, D_b=(0.04, 0.1))
    st = torch.cuda.Stream()

    def make():
        return mp.mp_init_batch(solid, u, Db, ka, kd, directions=directions, capacity=400, stream=st)
    own, ref, mixed = make(), make(), make()
    g = mp.mp_group_create([ref])
    plan = (1, 130, 7, 0, 62)
    for n in plan:
        mp.mp_step(own, n)
        mp.mp_group_step(g, n)
    g.close()
    for k, n in enumerate(plan):  # the group's steps and the context's own in turn
        if k % 2:
            h = mp.mp_group_create([mixed])
            mp.mp_group_step(h, n)
            h.close()
        else:
            mp.mp_step(mixed, n)
    for s in {0, species // 2, species - 1}:
        for f in range(1 + len(directions)):
            a = mp.mp_get_field(ref, s, f)
            for c in (own, mixed):
                b = mp.mp_get_field(c, s, f)
                assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])
        for d in directions:
            za, da = mp.mp_vacf(ref, s, "xyz".index(d))
            for c in (own, mixed):
                zb, db = mp.mp_vacf(c, s, "xyz".index(d))
                assert za.shape == zb.shape
                # FP64 sums of at most 1300 warp sums, each below |Z(0)|
                assert np.max(np.abs(za - zb)) <= 1e-12 * abs(za[0])
                assert np.max(np.abs(da - db)) <= 1e-10 * np.abs(da).max()
    for c in (own, ref, mixed):
        c.close()
