"""The series of a run of one step (appended by a launch of its own, from 6144 warps on over a cluster of
blocks) against the same steps in one run (appended by the next step, in one block): the same
Z and D bit for bit. Warp counts around the turns of the sums and the rule, several series."""
import numpy as np
import pytest

from paper_1303_2470_gb300 import media

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,directions,species,precision", [
    ((3, 3, 3), "x", 1, "fp32"), ((20, 20, 21), "xz", 1, "fp32"), ((32, 32, 33), "x", 1, "fp16"), ((63, 64, 65), "xyz", 1, "fp32"),
    ((64, 64, 65), "x", 3, "fp32"), ((64, 64, 48), "xy", 1, "fp32"), ((63, 65, 48), "z", 2, "fp16"),
    ((97, 64, 33), "x", 16, "fp32"), ((24, 33, 41), "xyz", 16, "fp32"), ((33, 31, 17), "xyz", 32, "fp16")])
def test_series_of_single_step_runs(shape, directions, species, precision):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1303_2470_gb300 import mp
    solid = media.bulk(*shape[::-1])
    solid[0, 0, 0] = 1
    u = torch.as_tensor(media.random_flow(solid, 0.01, seed=72).astype(np.float32)).cuda()
    Db, ka, kd = media.species(species, seed=73, D_b=(0.04, 0.1))
    a, b = (mp.mp_init_batch(solid, u, Db, ka, kd, directions=directions, precision=precision, capacity=20)
            for _ in range(2))
    mp.mp_step(a, 6)
    for n in (1, 1, 2, 1, 1):
        mp.mp_step(b, n)
    for s in range(species):
        for d in directions:
            (za, da), (zb, db) = (mp.mp_vacf(c, s, "xyz".index(d)) for c in (a, b))
            assert len(za) == 8 and np.array_equal(za, zb) and np.array_equal(da, db)
    a.close()
    b.close()
