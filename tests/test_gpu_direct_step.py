"""The one-launch-per-step kernel of the direct scheme at the edges of its forms: boxes as narrow as they
may be (every node near a wrap), and several species on either side of the sizes at which
one wave of 512, 768 or 1024 threads per SM takes the launch; the launch of one context against
the launch of several, with and without the link table.

Every form evaluates the same links in the same order with the same roundings, so fields are
bitwise equal; series are FP64 sums of the same per-warp FP32 sums in another order (1e-12). The
flux scheme differs by FP32 rounding: 2e-7 of the largest value per step at most (every term of a
step is rounded a few times at 6e-8), hence 1e-5 after 50 steps.
"""
import numpy as np
import pytest

from paper_1303_2470_gb300 import media

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _case(shape, species, seed):
    rng = np.random.default_rng(seed)
    solid = (rng.random(shape) < 0.35).astype(np.uint8)
    solid.flat[0] = 0
    u = (0.02 * rng.standard_normal((3,) + shape) * (solid == 0)).astype(np.float32)
    Db, ka, kd = media.species(species, seed=seed, D_b=(0.03, 0.08), k=(1e-3, 5e-2))
    return solid, torch.as_tensor(u).cuda(), Db, ka, kd


# fluid nodes (65 %): 88, 29, 91; 77 k and 79 k (152 SMs x 512 threads), 115 k and 119 k (768), 154 k and 158 k (1024)
@pytest.mark.parametrize("shape,species", [((9, 5, 3), 5), ((5, 3, 3), 3), ((7, 5, 4), 9), ((9, 5, 3), 1),
                                           ((40, 50, 59), 5), ((40, 50, 61), 5), ((50, 50, 71), 4), ((50, 50, 73), 4),
                                           ((60, 50, 79), 2), ((60, 50, 81), 2)])
def test_step_forms_agree(shape, species):
    from paper_1303_2470_gb300 import mp
    solid, u, Db, ka, kd = _case(shape, species, seed=sum(shape) + species)
    steps, dirs = 50, "xz"

    def make(**kw):
        return mp.mp_init_batch(solid, u, Db, ka, kd, directions=dirs, capacity=steps + 2, allow_negative=True, **kw)

    def result(ctx):
        fields = [f for s in range(species) for m in range(3) for f in mp.mp_get_field(ctx, s, m)]
        series = [x for s in range(species) for g in (0, 2) for x in mp.mp_vacf(ctx, s, g)]
        return fields, series

    ctxs = [make(scheme="direct", variant=v)
            for v in (0, mp.MP_VARIANT_RECOMPUTE, mp.MP_VARIANT_BLOCK128, mp.MP_VARIANT_PERSISTENT)]
    for c in ctxs:
        mp.mp_step(c, steps)
    pair = [make(scheme="direct") for _ in range(2)]
    mp.mp_group_step(mp.mp_group_create(pair), steps)
    flux = make(scheme="flux")
    mp.mp_step(flux, steps)
    F0, S0 = result(ctxs[0])
    for c in ctxs[1:] + pair:
        F, S = result(c)
        for a, b in zip(F0, F):
            assert np.array_equal(a, b)
        for a, b in zip(S0, S):
            assert np.max(np.abs(a - b)) <= 1e-12 * np.abs(a).max()
    F, S = result(flux)
    for a, b in zip(F0 + S0, F + S):
        assert np.max(np.abs(a - b)) <= 1e-5 * np.abs(b).max()
    for c in ctxs + pair + [flux]:
        c.close()
