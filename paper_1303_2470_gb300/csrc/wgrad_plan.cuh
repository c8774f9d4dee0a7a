// wgrad_plan.cuh -- shape of the tensor-core weight gradient (k_wgrad_tc in surrogate.cu) for one
// layer, and the order in which a block reuses its rings of staged rows (not part of the C ABI).
// Host and device, without CUDA headers, so that the bookkeeping also runs on the CPU.
#pragma once

#include <stddef.h>
#include <stdint.h>

#include <algorithm>

#ifdef __CUDACC__
#define MP_HOST_DEVICE __host__ __device__ __forceinline__
#else
#define MP_HOST_DEVICE inline
#endif

namespace mp {

constexpr int kColumn = 128;      // voxels of a column of work: 16 groups of 8 x-neighbours
constexpr int kColumnRows = 160;  // their staged rows: a group with its two neighbours is 10
constexpr int kBlockSmem = 232448 - 1024;  // dynamic shared memory a block may use (227 KB less static)
constexpr int kGStages = 8;       // most x stages

struct WgradPlan {
    int H;
    int GX, NG;          // groups per x-row, groups over the batch
    int T, nstrip;       // x rows per unit, strips along y
    int nci, nco, units;
    int nX;              // x stages; the dy ring has nX + 4 slots
    int bufs;            // accumulator sets
    uint32_t ncols;      // tensor-memory columns
    size_t smem;

    MP_HOST_DEVICE int combos() const { return 3 * nci * nco; }  // dz and channel blocks of a strip
    MP_HOST_DEVICE int slots() const { return nX + 4; }
    // x rows of unit u
    MP_HOST_DEVICE int rows(int u) const
    {
        const int left = H - u / combos() % nstrip * T;
        return T < left ? T : left;
    }
};

// x-rows are cut into groups of 8 voxels; the last one of a row may be short, and what it lacks
// is work done for nothing. Rows of one or two voxels (an eighth, a quarter of a group) stay with
// the tap-by-tap kernels, which the ones by columns beat by about three.
inline bool fills_groups(int W) { return W >= 3; }

inline int channel_block(int c) { return c % 64 == 0 ? 64 : (c % 32 == 0 ? 32 : 16); }

// Shape for one layer, or false where the kernel does not apply. T is the one with the least
// estimated time (waves of units x clocks of a unit, as in march_plan of surrogate.cu) that keeps
// a unit within 16 rows.
inline bool wgrad_plan(int B, int D, int H, int W, int Cin, int Cout, int sms, WgradPlan* m)
{
    if (!fills_groups(W) || (long long)B * D * H * W >= (1LL << 31)) return false;
    const int ci = channel_block(Cin), co = channel_block(Cout);
    const size_t xb = (size_t)kColumnRows * 2 * ci, yb = (size_t)kColumn * 2 * co;
    const int tiles = co == 64 ? 2 : 1, n = 3 * ci;
    // dy slots: the ring, two copies and what the padding rows of M read beyond a window
    const int pad = tiles * 128 / co - 1;
    int nX = kGStages;
    while (nX > 1 && nX * xb + (nX + 4 + pad) * yb > (size_t)kBlockSmem - 2048) --nX;
    if (nX < 2) return false;
    m->H = H;
    m->GX = (W + 7) / 8;
    m->NG = B * D * m->GX;
    m->nci = Cin / ci;
    m->nco = Cout / co;
    m->nX = nX;
    m->bufs = 2 * tiles * n <= 512 ? 2 : 1;
    m->ncols = 32;
    while ((int)m->ncols < m->bufs * tiles * n) m->ncols <<= 1;
    const double row = std::max(std::max(8.0 * tiles * std::max(n / 2.0, 32.0 + n / 4.0), (xb + yb) / 40.0), 300.0);
    const double flush = 12.0 * tiles * n;
    const long long per_row = (long long)m->combos() * ((m->NG + 15) / 16);
    double best = 0.0;
    for (int T = 1; T <= H && T <= 16; ++T) {
        const long long units = per_row * ((H + T - 1) / T);
        if (units > (1LL << 30)) continue;
        const double unit = std::max(T * row + 2.0 * yb / 40.0 + (m->bufs == 1 ? flush : 0.0), flush) + 500.0;
        const double cost = (double)((units + sms - 1) / sms) * unit + flush;
        if (best == 0.0 || cost < best) {
            best = cost;
            m->T = T;
            m->nstrip = (H + T - 1) / T;
            m->units = (int)units;
        }
    }
    m->smem = nX * xb + (nX + 4 + pad) * yb + 1024;
    return best > 0.0;
}

// What the copies of a block wait for beside the x slot (the stage nX back, which the slot was last
// used for). A stage is one x row; it reads three consecutive dy rows, and a unit of te x rows takes
// te + 2 dy rows: nX stages that belong to two units read nX + 4 dy rows, the dy ring's slots, but
// units shorter than nX - 1 rows put three and more units into nX stages. So a unit is copied
// only when the last but one before it has been read. Where units are long the x slot has seen
// to that, and nothing is waited for.
struct WgradUnits {
    int last = -1, before = -1;  // last stages of the unit before and of the one before that

    // the stage that has to be done before the first one of a unit, `stage`, is copied; -1: none
    // beside the x slot's (an older stage's barrier may be two phases on)
    MP_HOST_DEVICE int first_waits_for(const WgradPlan& p, int stage) const { return before > stage - p.nX ? before : -1; }
    MP_HOST_DEVICE void ended(int next_stage)
    {
        before = last;
        last = next_stage - 1;
    }
};

}  // namespace mp
