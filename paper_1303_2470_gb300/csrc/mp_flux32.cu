// mp_flux32.cu -- the flux-form step of mp.cu for contexts with FP32 arithmetic (FP32 or binary16
// storage) stepped on their own: the same update with the same roundings (see k_step there), so
// the fields are bitwise those of a grouped step.
//
// What bounds it: the L1 gathers of the sources and their latency (128^3, one species: L1 at 75 % of
// its rate, 53 % of the issue slots used, 677 instructions a node; the grouped body 725). What
// differs from that body:
//  * u*_g is tabulated (it depends on the flow only), which takes 30-60 instructions out of every
//    node and its accumulators out of the registers;
//  * no barrier: every warp stores its own partial sums (waiting for the block's slowest warp
//    was a quarter of all stall cycles), and the next launch appends the series in blocks of its
//    own instead of the last block of the step working alone;
//  * the per-species constants are read from the constant bank instead of shared memory;
//  * everything static is loaded before griddepcontrol.wait.
// Per step (the body of mp.cu -> this one): fcc 100^3 x 4 species 35.3 -> 16.7 us; 128^3 36.1 -> 26.1;
// 256^3 256 -> 200; 48^3 10.3 -> 5.8; 64^3 x 16 species x 2 moments 132 -> 64.6; binary16 88^3 x 2 moments
// 22.6 -> 14.7, 96^3 x 4 species 47.7 -> 26.1.
#include <cooperative_groups.h>

#include <algorithm>
#include <cstring>
#include <new>

#include "flux_run.cuh"
#include "internal.cuh"
#include "lattice.cuh"
#include "link_arith.cuh"
#include "mp_ctx.cuh"
#include "storage.cuh"

namespace mp {

struct F32Args {
    int nx, ny, nz, N, NF, NI, S, M, K;
    int chunks;  // 32-byte chunks of species (1 for one species)
    int nw;      // warps of nodes: NF / 32, rounded up
    int napp;    // blocks that append the series
    Div dx, dxy;
    const int32_t* flist;
    const uint32_t* fmask;
    const int32_t* aidx;      // compact interface index, -1 off the interface
    const Flow4<float>* u4;
    const float* ust;         // one species: [M][NF] u*_g; several: [2 M][NF] UA_g, UW_g
    double* part;             // [2][K][nw] the warps' partial sums of the series, by step parity
    // time index of the last appended step that read buffer 0 and 1. A step that reads buffer p
    // ends at time count[p] + 2: count[p] is written by the launch before it, never by its own.
    long long* count;
    double* Z;
    double* D;
    long long* tdev;
    long long cap;
    int stochastic;
    float whf[MP_MAX_SPECIES], whe[MP_MAX_SPECIES], hl[MP_MAX_SPECIES], pa[MP_MAX_SPECIES], pd[MP_MAX_SPECIES];
    double zsc[MP_MAX_SPECIES];
};

struct Flux32 {
    F32Args a;
    int32_t* aidx = nullptr;
    float* ust = nullptr;
    double* part = nullptr;
    long long* count = nullptr;
};

namespace {

constexpr uint32_t kAllLinks = (1u << 18) - 1u;
constexpr int kFinishBlocks = 8, kFinishThreads = 128;  // a series of k_finish32_wide

// appends the series of the step that read buffer `parity`: block b adds the series b, b + napp,
// ... over the warps (FP64, fixed order: four sums for each of kB threads; k_finish32_wide keeps to it)
template <int kB>
__device__ __forceinline__ void append32(const F32Args& a, int b, int parity)
{
    __shared__ double s_w[kB / 32];
    const long long t1 = *(volatile long long*)(a.count + (parity ^ 1)) + 1;
    for (int j = b; j < a.K; j += a.napp) {
        const double* p = a.part + ((size_t)parity * a.K + j) * a.nw;
        double v0 = 0.0, v1 = 0.0, v2 = 0.0, v3 = 0.0;
        int w = threadIdx.x;
        for (; w + 3 * kB < a.nw; w += 4 * kB) {
            v0 += __ldcg(p + w);
            v1 += __ldcg(p + w + kB);
            v2 += __ldcg(p + w + 2 * kB);
            v3 += __ldcg(p + w + 3 * kB);
        }
        for (; w < a.nw; w += kB) v0 += __ldcg(p + w);
        const double v = warp_sum((v0 + v1) + (v2 + v3));
        __syncthreads();
        if ((threadIdx.x & 31) == 0) s_w[threadIdx.x >> 5] = v;
        __syncthreads();
        if (threadIdx.x == 0) {
            double t = 0.0;
            for (int k = 0; k < kB / 32; ++k) t += s_w[k];
            const double z = t * a.zsc[j / a.M];
            a.Z[(size_t)j * a.cap + t1] = z;
            a.D[(size_t)j * a.cap + t1] = a.D[(size_t)j * a.cap + t1 - 1] + z;
        }
    }
    if (b == 0 && threadIdx.x == 0) {
        a.count[parity] = t1;
        *a.tdev = t1;
    }
}

// Blocks of 256, 6 per SM with one species (40 registers) and 3 with several (80). Measured per
// step, one species 128^3 / 256^3, 8 species 96^3, 16 species x 2 moments 64^3: 26.1 / 200 / 56.8 / 64.6 us;
// 5 and 2 blocks 27.4 / 219 / 65.4 / 88.8, 4 and 4 blocks 30.3 / 253 / 58.7 / 89.2, 8 blocks (32 registers) 26.3 /
// 196 but 48^3 7.1 (5.8), blocks of 128 x 12 and 5 26.3 / 225 / 58.0 / 95.2.
constexpr int kB = 256, kSingleBlocks = 6, kMultiBlocks = 3;

// blocks 0 .. napp-1 append the previous step, the others take kB nodes each. kCP: 32-byte chunks
// of species per pass of the link loop (0: one species)
template <typename TS, int FP, int kCP>
__global__ void __launch_bounds__(kB, kCP == 0 ? kSingleBlocks : kMultiBlocks)
    k_step32(const __grid_constant__ F32Args a, const TS* P_in, TS* __restrict__ Pn, const TS* A_in, TS* __restrict__ An,
             int parity, int pending)
{
    cudaTriggerProgrammaticLaunchCompletion();
    if ((int)blockIdx.x < a.napp) {
        cudaGridDependencySynchronize();
        if (pending) append32<kB>(a, blockIdx.x, parity ^ 1);
        return;
    }
    const int k = ((int)blockIdx.x - a.napp) * kB + (int)threadIdx.x;
    const int lane = threadIdx.x & 31;
    const bool active = k < a.NF;
    int n = 0, ai = -1;
    uint32_t mask = 0;
    Nbr b{};
    Flow4<float> ur{0.f, 0.f, 0.f, 0.f};
    if (active) {
        n = __ldg(a.flist + k);
        mask = __ldg(a.fmask + k);
        ai = __ldg(a.aidx + k);
        b = nbrs_of(a.nx, a.ny, a.nz, a.dx, a.dxy, n);
        ur = a.u4[n];
    }
    cudaGridDependencySynchronize();  // the previous step's fields, series and counts are visible
    const TS* P = after_wait(P_in);
    const TS* A = after_wait(A_in);
    // binary16 storage: rounding keys from the time index after this step, then array and element
    uint32_t tkey = 0;
    if constexpr (!std::is_same<float, TS>::value)
        tkey = hash32((uint32_t)(*(const volatile long long*)(a.count + parity) + 2));
    const uint32_t akey = tkey ^ 0x68e31da4u;
    double* part = a.part + (size_t)parity * a.K * a.nw + (k >> 5);  // series j: + j nw
    if constexpr (kCP == 0) {
        using V = FieldVec<float, FP>;
        using VS = FieldVec<TS, FP>;
        const VS* Pv = reinterpret_cast<const VS*>(P);
        float zv[3] = {0.f, 0.f, 0.f};
        if (active) {
            const V xr = ld_wide<float, TS, FP>(Pv + n);
            float delta[FP];
#pragma unroll
            for (int f = 0; f < FP; ++f) delta[f] = 0.f;
#pragma unroll
            for (int i = 1; i < kQ; ++i) {
                if ((mask >> (i - 1)) & 1u) {
                    const int s = src_of(b, i);
                    const Flow4<float> uf = a.u4[s];
                    const V xs = ld_wide<float, TS, FP>(Pv + s);
                    const float whl = is_face(i) ? a.whf[0] : a.whe[0];
                    const float pin =
                        rn_fma(weight<float>(i), qlink(edot<float>(i, uf.x, uf.y, uf.z), uf.w), whl);
                    const float pout =
                        rn_fma(weight<float>(i), qlink(edot<float>(opposite(i), ur.x, ur.y, ur.z), ur.w), whl);
#pragma unroll
                    for (int f = 0; f < FP; ++f)
                        delta[f] = rn_add(delta[f], rn_sub(rn_mul(pin, xs.v[f]), rn_mul(pout, xr.v[f])));
                }
            }
            float us[3];
#pragma unroll
            for (int m = 0; m < 3; ++m) us[m] = m < a.M ? __ldg(a.ust + (size_t)m * a.NF + k) : 0.f;
            V xan;
            if (ai >= 0) {
                const float pa = a.pa[0], pd = a.pd[0];
                const V xa = ld_wide<float, TS, FP>(reinterpret_cast<const VS*>(A) + ai);
#pragma unroll
                for (int f = 0; f < FP; ++f) {
                    const float js = rn_sub(rn_mul(pa, xr.v[f]), rn_mul(pd, xa.v[f]));
                    delta[f] = rn_sub(delta[f], js);
                    xan.v[f] = rn_add(xa.v[f], js);
                }
            }
            V xn;
#pragma unroll
            for (int f = 0; f < FP; ++f) xn.v[f] = rn_add(xr.v[f], delta[f]);
#pragma unroll
            for (int m = 0; m < 3; ++m)
                if (m < a.M && 1 + m < FP) zv[m] = xn.v[(1 + m) < FP ? 1 + m : 0] * us[m];
            if (ai >= 0)
                st_narrow<float, TS, FP>(reinterpret_cast<VS*>(An) + ai, xan, akey + (uint32_t)ai * FP, a.stochastic);
            st_narrow<float, TS, FP>(reinterpret_cast<VS*>(Pn) + n, xn, tkey + (uint32_t)n * FP, a.stochastic);
        }
#pragma unroll
        for (int m = 0; m < 3; ++m) {
            if (m < a.M) {
                const float w = warp_sum(zv[m]);
                if (lane == m && k - lane < a.NF) part[(size_t)m * a.nw] = (double)w;
            }
        }
    } else {
        constexpr int kSC = 8 / FP;
        constexpr int kMaxPass = kCP == 1 ? 1 : MP_MAX_SPECIES / (kCP * kSC);  // kCP 1: one chunk in all
        using VC = FieldVec<float, 8>;
        using VCS = FieldVec<TS, 8>;
        const VCS* Pc = reinterpret_cast<const VCS*>(P);
        VCS* __restrict__ Pnc = reinterpret_cast<VCS*>(Pn);
        const VCS* Ac = reinterpret_cast<const VCS*>(A);
        VCS* __restrict__ Anc = reinterpret_cast<VCS*>(An);
#pragma unroll
        for (int pass = 0; pass < kMaxPass; ++pass) {
            const int c0 = pass * kCP;
            if (c0 >= a.chunks) break;
            const int nc = a.chunks - c0 < kCP ? a.chunks - c0 : kCP;
            VC xr[kCP];
            float delta[kCP][8];
            if (active) {
#pragma unroll
                for (int cc = 0; cc < kCP; ++cc) {
                    if (cc < nc) xr[cc] = ld_wide<float, TS, 8>(Pc + (size_t)(c0 + cc) * a.N + n);
#pragma unroll
                    for (int j = 0; j < 8; ++j) delta[cc][j] = 0.f;
                }
#pragma unroll
                for (int i = 1; i < kQ; ++i) {
                    if ((mask >> (i - 1)) & 1u) {
                        const int s = src_of(b, i);
                        const Flow4<float> uf = a.u4[s];
                        const float qin = qlink(edot<float>(i, uf.x, uf.y, uf.z), uf.w);
                        const float qout = qlink(edot<float>(opposite(i), ur.x, ur.y, ur.z), ur.w);
#pragma unroll
                        for (int cc = 0; cc < kCP; ++cc) {
                            if (cc < nc) {
                                const VC xs = ld_wide<float, TS, 8>(Pc + (size_t)(c0 + cc) * a.N + s);
#pragma unroll
                                for (int q = 0; q < kSC; ++q) {
                                    const int sp = (c0 + cc) * kSC + q;
                                    const float whl = is_face(i) ? a.whf[sp] : a.whe[sp];
                                    const float pin = rn_fma(weight<float>(i), qin, whl);
                                    const float pout = rn_fma(weight<float>(i), qout, whl);
#pragma unroll
                                    for (int f = 0; f < FP; ++f) {
                                        const int j = q * FP + f;
                                        delta[cc][j] = rn_add(delta[cc][j],
                                                              rn_sub(rn_mul(pin, xs.v[j]), rn_mul(pout, xr[cc].v[j])));
                                    }
                                }
                            }
                        }
                    }
                }
            }
            // finish each chunk: sorption, Z terms, store, warp sums of the Z terms
            float UA[3], UW[3];
#pragma unroll
            for (int m = 0; m < 3; ++m) {
                const bool on = active && m < a.M;
                UA[m] = on ? __ldg(a.ust + (size_t)(2 * m) * a.NF + k) : 0.f;
                UW[m] = on ? __ldg(a.ust + (size_t)(2 * m + 1) * a.NF + k) : 0.f;
            }
#pragma unroll
            for (int cc = 0; cc < kCP; ++cc) {
                float zv[kSC][3];
#pragma unroll
                for (int q = 0; q < kSC; ++q)
#pragma unroll
                    for (int m = 0; m < 3; ++m) zv[q][m] = 0.f;
                if (active && cc < nc) {
                    if (ai >= 0) {
                        const size_t ia = (size_t)(c0 + cc) * a.NI + ai;
                        const VC xa = ld_wide<float, TS, 8>(Ac + ia);
                        VC xan;
#pragma unroll
                        for (int q = 0; q < kSC; ++q) {
                            const int sp = (c0 + cc) * kSC + q;
                            const float pa = a.pa[sp], pd = a.pd[sp];
#pragma unroll
                            for (int f = 0; f < FP; ++f) {
                                const int j = q * FP + f;
                                const float js = rn_sub(rn_mul(pa, xr[cc].v[j]), rn_mul(pd, xa.v[j]));
                                delta[cc][j] = rn_sub(delta[cc][j], js);
                                xan.v[j] = rn_add(xa.v[j], js);
                            }
                        }
                        st_narrow<float, TS, 8>(Anc + ia, xan, akey + (uint32_t)ia * 8, a.stochastic);
                    }
                    VC xn;
#pragma unroll
                    for (int j = 0; j < 8; ++j) xn.v[j] = rn_add(xr[cc].v[j], delta[cc][j]);
                    const size_t pi = (size_t)(c0 + cc) * a.N + n;
                    st_narrow<float, TS, 8>(Pnc + pi, xn, tkey + (uint32_t)pi * 8, a.stochastic);
#pragma unroll
                    for (int q = 0; q < kSC; ++q) {
                        const float h = a.hl[(c0 + cc) * kSC + q];
#pragma unroll
                        for (int m = 0; m < 3; ++m)
                            if (m < a.M && 1 + m < FP)
                                zv[q][m] = xn.v[q * FP + ((1 + m) < FP ? 1 + m : 0)] * (UA[m] + h * UW[m]);
                    }
                }
#pragma unroll
                for (int q = 0; q < kSC; ++q) {
                    const int sp = (c0 + cc) * kSC + q;
                    if (cc < nc && sp < a.S) {
#pragma unroll
                        for (int m = 0; m < 3; ++m) {
                            if (m < a.M) {
                                const float w = warp_sum(zv[q][m]);
                                if (lane == 0 && k < a.NF) part[(size_t)(sp * a.M + m) * a.nw] = (double)w;
                            }
                        }
                    }
                }
            }
        }
    }
}

// append32 as a launch of its own (the last step of a run)
__global__ void __launch_bounds__(kB) k_finish32(const __grid_constant__ F32Args a, int parity)
{
    pdl_enter();
    append32<kB>(a, blockIdx.x, parity);
}

// The same where the series are sums of many warps (kWideSeries and more): nothing hides this launch,
// and one SM adds two FP64 numbers a clock. The four sums of append32's kB threads are spread over the
// blocks of a cluster, one sum a thread, and put together in the same order in the first block's
// shared memory. Runs of one step, one block a series / a cluster: 64^3 (3.3 k warps) 12.6 / 13.3 us,
// 128^3 (26 k) 42.0 / 36.3, 256^3 (210 k) 327 / 240.
constexpr int kWideSeries = 6144;
__global__ void __cluster_dims__(kFinishBlocks, 1, 1) __launch_bounds__(kFinishThreads)
    k_finish32_wide(const __grid_constant__ F32Args a, int parity)
{
    static_assert(kFinishBlocks * kFinishThreads == 4 * kB, "one sum a thread");
    namespace cg = cooperative_groups;
    __shared__ double s_v[4 * kB];
    __shared__ double s_w[kB / 32];
    const cg::cluster_group cluster = cg::this_cluster();
    const int rank = (int)cluster.block_rank(), b = (int)blockIdx.x / kFinishBlocks;
    double* sums = cluster.map_shared_rank(s_v, 0);
    pdl_enter();
    const long long t1 = *(volatile long long*)(a.count + (parity ^ 1)) + 1;
    const int q = rank * kFinishThreads + (int)threadIdx.x, first = q % kB, col = q / kB * kB;
    for (int j = b; j < a.K; j += a.napp) {
        const double* p = a.part + ((size_t)parity * a.K + j) * a.nw;
        double v = 0.0;
        int w = first;
        for (; w + 28 * kB + 3 * kB < a.nw; w += 32 * kB) {
            double x[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) x[k] = __ldcg(p + w + col + 4 * k * kB);
#pragma unroll
            for (int k = 0; k < 8; ++k) v += x[k];
        }
        for (; w + 3 * kB < a.nw; w += 4 * kB) v += __ldcg(p + w + col);
        if (col == 0)
            for (; w < a.nw; w += kB) v += __ldcg(p + w);
        sums[q] = v;
        cluster.sync();
        if (rank == 0) {
#pragma unroll
            for (int i = (int)threadIdx.x; i < kB; i += kFinishThreads) {
                const double u = warp_sum((s_v[i] + s_v[i + kB]) + (s_v[i + 2 * kB] + s_v[i + 3 * kB]));
                if ((i & 31) == 0) s_w[i >> 5] = u;
            }
            __syncthreads();
            if (threadIdx.x == 0) {
                double t = 0.0;
                for (int k = 0; k < kB / 32; ++k) t += s_w[k];
                const double z = t * a.zsc[j / a.M];
                a.Z[(size_t)j * a.cap + t1] = z;
                a.D[(size_t)j * a.cap + t1] = a.D[(size_t)j * a.cap + t1 - 1] + z;
            }
        }
        cluster.sync();  // the first block's sums are free again, and stay until every block has written
    }
    if (q == 0 && b == 0) {
        a.count[parity] = t1;
        *a.tdev = t1;
    }
}

// counts from the series position (after other launches have moved it): next: the buffer that the
// next step reads
__global__ void k_counts32(const F32Args a, int next)
{
    const long long t = *a.tdev;
    a.count[next] = t - 1;
    a.count[next ^ 1] = t;
}

// interface indices and the flow-dependent sums of u*_g, added in the order of the step of mp.cu
__global__ void k_tables32(const F32Args a, const uint32_t* __restrict__ iface, const int32_t* __restrict__ ibase, int d0,
                           int d1, int d2, int32_t* __restrict__ aidx, float* __restrict__ ust)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= a.NF) return;
    const int n = a.flist[k];
    const uint32_t mask = a.fmask[k];
    aidx[k] = mask != kAllLinks ? ibase[n >> 5] + __popc(iface[n >> 5] & ((1u << (n & 31)) - 1u)) : -1;
    const Flow4<float> ur = a.u4[n];
    const int dir[3] = {d0, d1, d2};
    for (int m = 0; m < a.M; ++m) {
        const int g = dir[m];
        float us = 0.f, ua = 0.f, uw = 0.f;
#pragma unroll
        for (int i = 1; i < kQ; ++i) {
            if (!((mask >> (i - 1)) & 1u)) continue;
            const int c = g == 0 ? cx(opposite(i)) : (g == 1 ? cy(opposite(i)) : cz(opposite(i)));
            const float qout = qlink(edot<float>(opposite(i), ur.x, ur.y, ur.z), ur.w);
            if (c != 0) {
                us += (float)c * rn_fma(weight<float>(i), qout, is_face(i) ? a.whf[0] : a.whe[0]);
                ua = fmaf((float)c * weight<float>(i), qout, ua);
                uw += (float)c * weight<float>(i);
            }
        }
        if (a.S == 1) {
            ust[(size_t)m * a.NF + k] = us;
        } else {
            ust[(size_t)(2 * m) * a.NF + k] = ua;
            ust[(size_t)(2 * m + 1) * a.NF + k] = uw;
        }
    }
}

template <typename TS>
int step32(mp_ctx* c, long long n)
{
    const F32Args& a = c->flux32->a;
    auto kern = c->FP == 2 ? (c->S == 1 ? k_step32<TS, 2, 0> : (a.chunks == 1 ? k_step32<TS, 2, 1> : k_step32<TS, 2, 2>))
                           : (c->S == 1 ? k_step32<TS, 4, 0> : (a.chunks == 1 ? k_step32<TS, 4, 1> : k_step32<TS, 4, 2>));
    const int blocks = a.napp + (a.NF + kB - 1) / kB;
    return run_flux(
        c, n,
        [&](int pending, bool programmatic) {
            const int s = c->cur;
            return launch_dependent(programmatic, kern, dim3(blocks), dim3(kB), c->stream, a, (const TS*)c->P[s],
                                    (TS*)c->P[1 - s], (const TS*)c->A[s], (TS*)c->A[1 - s], s, pending);
        },
        [&](int parity) {
            return a.nw < kWideSeries
                       ? launch_pdl(k_finish32, dim3(a.napp), dim3(kB), c->stream, a, parity)
                       : launch_pdl(k_finish32_wide, dim3(kFinishBlocks * a.napp), dim3(kFinishThreads), c->stream, a, parity);
        });
}

}  // namespace

void flux32_free(mp_ctx* c)
{
    if (!c->flux32) return;
    cudaFree(c->flux32->aidx);
    cudaFree(c->flux32->ust);
    cudaFree(c->flux32->part);
    cudaFree(c->flux32->count);
    delete c->flux32;
    c->flux32 = nullptr;
}

// Tables: 4 bytes per fluid node and 4 (one species) or 8 per direction, and half a byte per series;
// where they do not fit (tables_fit) or cannot be allocated the context keeps the step of mp.cu
// (c->flux32 stays NULL).
int flux32_setup(mp_ctx* c)
{
    const size_t NF = (size_t)c->geo.n_fluid, K = (size_t)(c->S * c->M);
    const size_t nw = (NF + 31) / 32;  // warps of nodes
    const size_t ust_bytes = sizeof(float) * (c->S == 1 ? 1 : 2) * (size_t)c->M * NF, part_bytes = sizeof(double) * 2 * K * nw;
    if (!tables_fit(sizeof(int32_t) * NF + ust_bytes + part_bytes)) return MP_OK;
    Flux32* f = new (std::nothrow) Flux32();
    if (!f) return MP_OK;
    c->flux32 = f;
    F32Args& a = f->a;
    memset(&a, 0, sizeof(a));
    a.nx = c->geo.nx;
    a.ny = c->geo.ny;
    a.nz = c->geo.nz;
    a.N = c->geo.N;
    a.NF = (int)NF;
    a.NI = (int)c->geo.n_iface;
    a.S = c->S;
    a.M = c->M;
    a.K = (int)K;
    a.chunks = c->S == 1 ? 1 : c->SP / c->SC;
    a.nw = (int)nw;
    a.napp = (int)std::min<size_t>(K, 64);
    a.dx = make_div((unsigned)c->geo.nx);
    a.dxy = make_div((unsigned)(c->geo.nx * c->geo.ny));
    cudaError_t e = cudaMalloc(&f->aidx, sizeof(int32_t) * NF);
    if (e == cudaSuccess) e = cudaMalloc(&f->ust, ust_bytes);
    if (e == cudaSuccess) e = cudaMalloc(&f->part, part_bytes);
    if (e == cudaSuccess) e = cudaMalloc(&f->count, sizeof(long long) * 2);
    if (e != cudaSuccess) {
        (void)cudaGetLastError();
        flux32_free(c);
        return MP_OK;
    }
    a.flist = c->geo.flist;
    a.fmask = c->fmask;
    a.aidx = f->aidx;
    a.u4 = (const Flow4<float>*)c->u4;
    a.ust = f->ust;
    a.part = f->part;
    a.count = f->count;
    a.Z = c->Z;
    a.D = c->D;
    a.tdev = c->tdev;
    a.cap = c->cap;
    a.stochastic = c->stochastic;
    for (int s = 0; s < c->S; ++s) {
        a.hl[s] = (float)(6.0 * c->Db[s]);  // lambda/2 = 12 D_b / 2
        a.whf[s] = (float)((double)weight<float>(1) * (double)a.hl[s]);
        a.whe[s] = (float)((double)weight<float>(5) * (double)a.hl[s]);
        a.pa[s] = (float)c->ka[s];
        a.pd[s] = (float)c->kd[s];
    }
    for (int s = 0; s < c->S; ++s) a.zsc[s] = c->zsc[s];
    k_tables32<<<(unsigned)((NF + 255) / 256), 256, 0, c->stream>>>(a, c->geo.iface, c->geo.ibase, c->dir[0], c->dir[1],
                                                                    c->dir[2], f->aidx, f->ust);
    MP_CUDA(cudaGetLastError());
    c->series_moved = true;
    c->tables_new = true;
    return MP_OK;
}

int flux32_step(mp_ctx* c, long long n)
{
    if (n <= 0) return MP_OK;
    if (c->series_moved) {
        k_counts32<<<1, 1, 0, c->stream>>>(c->flux32->a, c->cur);
        MP_CUDA(cudaGetLastError());
        c->series_moved = false;
    }
    return c->precision == MP_FP16 ? step32<__half>(c, n) : step32<float>(c, n);
}

}  // namespace mp
