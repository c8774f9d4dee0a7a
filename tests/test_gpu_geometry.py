"""Node classes and the largest cluster beyond one block of the prefix scan (1024 words of 32
nodes), with ragged last words, clusters that meet only through the periodic faces, a long
winding channel and equal clusters (the one with the smallest node wins). Everything is whole
numbers: equal to the oracle's classes and largest cluster."""
import numpy as np
import pytest

import oracle
from paper_1303_2470_gb300 import media

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _serpentine(nx, ny, nz):
    """One channel of single nodes winding through a plane: every second row, joined at
    alternating ends."""
    s = np.ones((nz, ny, nx), dtype=np.uint8)
    for j, y in enumerate(range(1, ny - 1, 3)):
        s[nz // 2, y, 1:nx - 1] = 0
        if y + 3 < ny - 1:
            x = nx - 2 if j % 2 == 0 else 1
            s[nz // 2, y:y + 4, x] = 0
    return s


def _media():
    rng = np.random.default_rng(5)
    yield np.zeros((3, 3, 3), dtype=np.uint8)
    yield np.ones((4, 5, 6), dtype=np.uint8)
    yield (rng.random((5, 7, 33)) < 0.9).astype(np.uint8)
    yield media.random_spheres((41, 40, 43), 4, 0.3, seed=6)[0]
    yield (rng.random((37, 39, 41)) < 0.92).astype(np.uint8)       # thousands of small clusters
    yield (np.indices((33, 34, 36)).sum(0) % 2).astype(np.uint8)   # links along edges only
    yield _serpentine(61, 130, 9)
    two = np.ones((12, 40, 70), dtype=np.uint8)                    # equal clusters; one across the faces
    two[3, 10, 5:25] = 0
    two[9, 30, 60:] = 0
    two[9, 30, :10] = 0
    yield two


@pytest.mark.parametrize("k", range(8))
def test_classes_and_largest_cluster(k):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1303_2470_gb300 import mp
    solid = list(_media())[k]
    ocls, onf, oni = oracle.classify(solid)
    big = oracle.largest_cluster(solid)[0].astype(bool) if onf else np.zeros(solid.shape, bool)
    want = (ocls + 4 * big).astype(np.uint8)
    for arg in (solid, torch.as_tensor(solid).cuda()):
        cls, (nf, ni, nc) = mp.mp_classify(arg)
        assert (nf, ni, nc) == (onf, oni, int(big.sum()))
        assert np.array_equal(cls, want)
        for off in (0, 1):
            buf = torch.full((solid.size + 8,), 77, dtype=torch.uint8, device="cuda")
            out = buf[off:off + solid.size]
            assert mp.mp_classify_device(arg, out) == (onf, oni)
            assert np.array_equal(out.cpu().numpy().reshape(solid.shape), want)
            assert int(buf[off + solid.size]) == 77
    mp.mp_release_cached()
    assert mp.mp_classify(solid)[1] == (onf, oni, int(big.sum()))
