"""The quick path of mp_step_noalloc's binding takes the scalar arguments that the general path
takes (both convert them). CPU: the library's function is replaced by one of the same argument
types that records what arrives."""
import ctypes
import types

import numpy as np
import pytest
import torch


@pytest.mark.parametrize("D_b,direction", [(0.05, 1), (0.05, 1.0), (np.float64(0.05), np.float32(1)), ("0.05", "1"),
                                           (np.float32(0.05), np.int64(1)), (torch.tensor(0.05), torch.tensor(1.0))])
def test_quick_path_converts_its_scalars(monkeypatch, D_b, direction):
    from paper_1303_2470_gb300 import build
    build.build()
    from paper_1303_2470_gb300 import mp
    got = []
    call = ctypes.CFUNCTYPE(ctypes.c_int, *mp._lib.mp_step_noalloc.argtypes)(lambda *a: got.append(a) or 0)
    monkeypatch.setattr(mp, "_lib", types.SimpleNamespace(mp_step_noalloc=call))
    monkeypatch.setattr(mp, "_noalloc_device", lambda *a: 0)
    monkeypatch.setattr(torch.cuda, "current_device", lambda: 0)
    solid = torch.zeros((4, 5, 6), dtype=torch.uint8)
    f = [torch.zeros((4, 5, 6)) for _ in range(4)]
    mp.mp_step_noalloc(solid, None, D_b, 0, np.float64(0.5), direction, *f, torch.zeros(1, dtype=torch.float64))
    assert len(got) == 1
    assert got[0][:3] == (6, 5, 4) and got[0][5] == pytest.approx(0.05) and got[0][6:9] == (0.0, 0.5, 1)
