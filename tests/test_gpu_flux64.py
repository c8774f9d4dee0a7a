"""The tabulated FP64 flux step at the edges of its launch forms: four lanes a node up to
19456 fluid nodes, one (density + one moment) or two (more moments) beyond, a last group of
32 nodes and a last block that are not full, one and several species. Against the FP64
oracle; tolerance as for every FP64 comparison here: 60 steps of order-1 sums in FP64."""
import numpy as np
import pytest

import oracle
from paper_1303_2470_gb300 import media

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,directions,species", [
    ((3, 3, 3), "x", 1),          # fewer nodes than a block
    ((5, 7, 9), "xyz", 3),
    ((29, 31, 33), "x", 1),       # beyond 19456 nodes: one lane a node
    ((31, 29, 33), "z", 2),
    ((33, 31, 29), "xz", 1),      # two lanes a node
    ((33, 29, 31), "xyz", 3),
])
def test_fp64_step_matches_oracle(shape, directions, species):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1303_2470_gb300 import mp
    solid, _ = media.random_spheres(shape, 1 if max(shape) < 9 else 2, 0.8, seed=31)
    u = media.random_flow(solid, 0.01, seed=32).astype(np.float32)
    Db, ka, kd = media.species(species, seed=33, D_b=(0.04, 0.1))
    big = int((solid == 0).sum()) > 152 * 16 * 8
    assert big == (max(shape) > 9)
    steps = 60
    for stream in (None, torch.cuda.Stream()):
        ctx = mp.mp_init_batch(solid, torch.as_tensor(u).cuda(), Db, ka, kd, precision="fp64", directions=directions,
                               capacity=steps + 2, stream=stream)
        mp.mp_step(ctx, 1)
        mp.mp_step(ctx, 0)
        mp.mp_step(ctx, steps - 1)
        for s in range(species):
            p = oracle.Problem(solid, u.astype(np.float64), Db[s], ka[s], kd[s])
            for d in directions:
                Z, D = mp.mp_vacf(ctx, s, "xyz".index(d))
                ref = oracle.run(p, g="xyz".index(d), nsteps=steps)
                assert np.max(np.abs(Z - ref.Z)) < 1e-11 * abs(ref.Z[0])
                assert np.max(np.abs(D - ref.D)) < 1e-11 * np.abs(ref.D).max()
            m = mp.mp_mass(ctx, s)
            assert abs(m[0] + m[1] - 1.0) < 1e-11
        ctx.close()
