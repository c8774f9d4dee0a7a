"""A step reads its tables before it waits for the launch before it, so the first step after set-up
must not be a programmatic dependent launch. The launches of run_flux are recorded on the CPU with the
header that the library uses; on the GPU, first steps right behind the set-up are compared
with first steps after a synchronisation."""
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
RECORD = r"""
#include <cstdio>
#include "flux_run.cuh"
namespace mp {
int cuda_fail(cudaError_t, const char*) { return MP_OK; }  // no device here
}
int main()
{
    mp_ctx c;                // the default stream: no graph
    c.tables_new = true;     // as the set-up leaves it
    for (int n : {0, 3, 2}) {
        mp::run_flux(
            &c, n,
            [&](int pending, bool programmatic) {
                std::printf("step%d%d ", pending, (int)programmatic);
                return cudaSuccess;
            },
            [&](int) {
                std::printf("finish ");
                return cudaSuccess;
            });
        std::printf("| ");
    }
    std::printf("t=%lld\n", c.t);
}
"""


def test_first_step_after_set_up_is_an_ordinary_launch(tmp_path):
    from paper_1303_2470_gb300 import build
    (tmp_path / "record.cu").write_text(RECORD)
    exe = tmp_path / "record"
    subprocess.run([build._nvcc(), "-std=c++17", "-I", os.path.join(ROOT, "paper_1303_2470_gb300", "csrc"),
                    str(tmp_path / "record.cu"), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout
    assert out == "| step00 step11 step11 finish | step01 step11 finish | t=5\n"


@pytest.mark.gpu
@pytest.mark.parametrize("precision,species", [("fp64", 1), ("fp64", 3), ("fp32", 1), ("fp16", 4)])
@pytest.mark.parametrize("shape", [(3, 4, 5), (61, 53, 47)])
def test_first_steps_right_behind_the_set_up(precision, species, shape):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1303_2470_gb300 import media, mp
    solid, _ = media.random_spheres(shape, 1 if max(shape) < 9 else 3, 0.8, seed=51)
    u = torch.as_tensor(media.random_flow(solid, 0.01, seed=52).astype(np.float32)).cuda()
    Db, ka, kd = media.species(species, seed=53, D_b=(0.04, 0.1))
    for stream in (None, torch.cuda.Stream()):
        torch.cuda.synchronize()
        got = []
        for wait in (True, False, False, False):
            ctx = mp.mp_init_batch(solid, u, Db, ka, kd, precision=precision, capacity=8, stream=stream)
            if wait:
                torch.cuda.synchronize()
            mp.mp_step(ctx, 1)
            mp.mp_step(ctx, 2)
            got.append([mp.mp_get_field(ctx, s, 1) for s in range(species)] + [mp.mp_vacf(ctx, 0, 0)])
            ctx.close()
        for other in got[1:]:
            for a, b in zip(got[0], other):
                assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])
