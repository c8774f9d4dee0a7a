"""Flux contexts with and without their step tables: the rule that leaves them out (CPU), and the
step that recomputes what they hold against the one that reads them (GPU): the same fields bit for bit
with FP32 and binary16 storage; Z, D and FP64 fields up to the order of FP64 sums (at most 20
terms a node and step, 200 steps, so 1e-12 of the largest value)."""
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
RULE = r"""
#include <cstdio>
#include "flux_run.cuh"
namespace mp {
int cuda_fail(cudaError_t, const char*) { return MP_OK; }
}
int main()
{
    const size_t mb = 1 << 20;
    std::printf("%d%d%d%d%d\n", mp::tables_fit(64 * mb, 0), mp::tables_fit(64 * mb + 1, 0), mp::tables_fit(100 * mb, 400 * mb),
                mp::tables_fit(100 * mb, 400 * mb - 4), mp::tables_fit(100000 * mb, 280000 * mb));
}
"""


def test_rule_for_the_tables(tmp_path):
    from paper_1303_2470_gb300 import build
    (tmp_path / "rule.cu").write_text(RULE)
    exe = tmp_path / "rule"
    subprocess.run([build._nvcc(), "-std=c++17", "-I", os.path.join(ROOT, "paper_1303_2470_gb300", "csrc"),
                    str(tmp_path / "rule.cu"), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout == "10100\n"


@pytest.mark.gpu
@pytest.mark.parametrize("precision", ["fp32", "fp16", "fp64"])
@pytest.mark.parametrize("shape,directions,species", [((3, 3, 4), "x", 1), ((9, 11, 13), "xyz", 1), ((8, 9, 10), "y", 5),
                                                      ((13, 12, 11), "xz", 3)])
def test_steps_without_tables(precision, shape, directions, species):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1303_2470_gb300 import media, mp
    solid = media.bulk(*shape[::-1]) if min(shape) < 4 else media.random_spheres(shape, 2, 0.7, seed=61)[0]
    u = torch.as_tensor(media.random_flow(solid, 0.01, seed=62).astype(np.float32)).cuda()
    Db, ka, kd = media.species(species, seed=63, D_b=(0.04, 0.1))
    for stream in (None, torch.cuda.Stream()):
        torch.cuda.synchronize()
        ctxs = [mp.mp_init_batch(solid, u, Db, ka, kd, precision=precision, directions=directions, capacity=300,
                                 stream=stream, variant=v) for v in (0, 1)]
        for n in (1, 130, 7, 0, 62):
            for c in ctxs:
                mp.mp_step(c, n)
        for s in range(species):
            for f in range(1 + len(directions)):
                (a, aa), (b, bb) = (mp.mp_get_field(c, s, f) for c in ctxs)
                if precision == "fp64":
                    assert np.max(np.abs(a - b)) <= 1e-12 * np.abs(a).max()
                    assert np.max(np.abs(aa - bb)) <= 1e-12 * max(np.abs(aa).max(), np.abs(a).max())
                else:
                    assert np.array_equal(a, b) and np.array_equal(aa, bb)
            for d in directions:
                (za, da), (zb, db) = (mp.mp_vacf(c, s, "xyz".index(d)) for c in ctxs)
                assert np.max(np.abs(za - zb)) <= 1e-12 * abs(za[0])
                assert np.max(np.abs(da - db)) <= 1e-10 * np.abs(da).max()
        for c in ctxs:
            c.close()
