"""The rings of staged rows of the tensor-core weight gradient, replayed on the CPU with the header
that the kernel uses (csrc/wgrad_plan.cuh): every block's copies in order, and its MMAs as late as the
waits allow (a stage is read only when a copy waits for it). Each stage must then still find its x row
and its three dy rows in the slots that the kernel's descriptors start from."""
import ctypes
import os
import random
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
REPLAY = r"""
#include <vector>
#include "wgrad_plan.cuh"
using namespace mp;

// rows read wrongly (2^30: a wait for a stage not yet copied, or for a barrier that may be two
// phases on); -1: no plan. out: T, units, x stages, and the most units that one block's last
// nX stages belonged to
extern "C" int replay(int B, int D, int H, int W, int Cin, int Cout, int sms, int* out)
{
    WgradPlan p;
    if (!wgrad_plan(B, D, H, W, Cin, Cout, sms, &p)) return -1;
    const int step = std::min(p.units, sms), R = p.slots();
    int wrong = 0, most = 0;
    for (int block = 0; block < step; ++block) {
        std::vector<int> x(p.nX, -1), y(R + 2, -1);
        std::vector<int> first, number;  // each copied stage's first dy row, and its unit's number in the block
        WgradUnits units;
        int stage = 0, ys = 0, next_y = 0, n = 0, read = 0;
        auto mma_to = [&](int last) {  // as k_wgrad_tc's MMA warp: the slots follow from the rows alone
            for (; read <= last; ++read) {
                const int at = first[read] % R;
                wrong += x[read % p.nX] != read;
                for (int k = 0; k < 3; ++k) wrong += y[at + k] != first[read] + k;
            }
        };
        auto load_y = [&] {
            y[ys] = next_y;
            if (ys < 2) y[ys + R] = next_y;
            ++next_y;
            ys = ys + 1 == R ? 0 : ys + 1;
        };
        for (int u = block; u < p.units; u += step, ++n) {
            const int te = p.rows(u), start = stage;
            const int w = units.first_waits_for(p, start);
            if (w >= start || (w >= 0 && w <= start - p.nX)) return 1 << 30;
            for (int i = 0; i < te; ++i, ++stage) {
                mma_to(stage - p.nX);
                if (i == 0) {
                    if (w >= 0) mma_to(w);
                    load_y();
                    load_y();
                }
                load_y();
                x[stage % p.nX] = stage;
                first.push_back(start + 2 * n + i);
                number.push_back(n);
                most = std::max(most, n - number[std::max(0, stage - p.nX + 1)] + 1);
            }
            units.ended(stage);
        }
        mma_to(stage - 1);
    }
    out[0] = p.T;
    out[1] = p.units;
    out[2] = p.nX;
    out[3] = most;
    return wrong;
}
"""
CHANNELS = [(16, 32), (32, 32), (32, 64), (64, 64), (64, 96), (96, 96), (96, 128), (128, 128), (128, 96), (96, 64),
            (64, 32), (32, 16), (16, 16), (48, 272)]


@pytest.fixture(scope="module")
def replay(tmp_path_factory):
    d = tmp_path_factory.mktemp("ring")
    (d / "replay.cpp").write_text(REPLAY)
    so = d / "replay.so"
    subprocess.run(["g++", "-std=c++17", "-O2", "-Wall", "-Werror", "-shared", "-fPIC", "-I",
                    os.path.join(ROOT, "paper_1303_2470_gb300", "csrc"), str(d / "replay.cpp"), "-o", str(so)], check=True)
    lib = ctypes.CDLL(str(so))

    def call(*shape, sms=152):
        out = (ctypes.c_int * 4)()
        return lib.replay(*shape, sms, out), list(out)
    return call


@pytest.mark.parametrize("sms", [152, 148, 7])
def test_short_units_keep_unread_rows(replay, sms):
    """Layers whose units are shorter than the rings, so that nX stages touch three units and more:
    the levels of 48^3 and 64^3 training boxes, and short last strips."""
    deepest = 0
    for shape in [(4, 12, 12, 12, 96, 96), (4, 12, 12, 12, 128, 96), (1, 48, 48, 48, 32, 32), (1, 48, 48, 48, 32, 16),
                  (2, 16, 16, 16, 96, 96), (3, 16, 16, 16, 128, 96), (4, 18, 7, 118, 32, 16), (4, 64, 4, 128, 32, 32),
                  (2, 24, 1, 40, 64, 64), (1, 9, 33, 64, 16, 16), (3, 20, 17, 30, 64, 32)]:
        wrong, (_, _, _, most) = replay(*shape, sms=sms)
        assert wrong == 0, shape
        deepest = max(deepest, most)
    assert deepest >= 3  # the case that a ring of nX + 4 rows has no room for


def test_layers_over_the_range(replay):
    rng = random.Random(5)
    for _ in range(400):
        K, N = rng.choice(CHANNELS)
        shape = (rng.randint(1, 4), rng.randint(1, 24), rng.randint(1, 64), rng.randint(3, 128), K, N)
        wrong, _ = replay(*shape, sms=rng.choice([152, 148, 20, 3]))
        assert wrong == 0, shape
