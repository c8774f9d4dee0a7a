// surrogate.cu -- kernels of the learned warm start for lb_steady (include/surrogate.h): 3x3x3
// periodic convolutions, forward and both gradients, on the 5th-generation tensor cores
// (tcgen05.mma with accumulators in tensor memory; the weight gradient of boxes narrower than three
// voxels or of very few with mma.sync m16n8k16; BF16 operands, FP32 accumulation),
// pooling, upsampling, the masked loss and the Adam update. Nothing here belongs to the moment-propagation
// method itself; the network's output only seeds lb_steady.
#include <algorithm>

#include <cuda.h>
#include <cuda_bf16.h>

#include "../../include/surrogate.h"
#include "internal.cuh"
#include "wgrad_plan.cuh"

using namespace mp;

namespace {

typedef __nv_bfloat16 bf16;

__device__ __forceinline__ int wrap(int v, int n) { return v < 0 ? v + n : (v >= n ? v - n : v); }

// D += A B for one m16n8k16 tile; fragments as the PTX ISA lays them out for .bf16:
// a0..a3 rows (g, g+8) x cols (2t, 2t+1) and (+8); b0, b1 rows (2t, 2t+1) and (+8) of col g.
__device__ __forceinline__ void mma16816(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                         uint32_t b0, uint32_t b1)
{
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

struct ConvArgs {
    const bf16* x;
    const bf16* w;
    const float* bias;
    bf16* y;
    float* yf;
    int D, H, W, V, K, N, sign, relu;
    // second BF16 output, from y = act(...) rounded to BF16 and `other` [B][V][N]: y + other
    // (mode 1), or (kMask) y where other > 0, else 0
    bf16* y2;
    const bf16* other;
    int mode;
    int up;  // x is the coarse grid [B][D/2][H/2][W/2][K], read as its nearest upsampling
};
constexpr int kMask = 2;

// voxel of the stored x that fine voxel (b, z, y, x) of a D x H x W box reads
__device__ __forceinline__ int x_voxel(int up, int D, int H, int W, int b, int z, int y, int x)
{
    return up ? ((b * (D >> 1) + (z >> 1)) * (H >> 1) + (y >> 1)) * (W >> 1) + (x >> 1)
              : ((b * D + z) * H + y) * W + x;
}

// eight BF16 values as FP32 and back
__device__ __forceinline__ void unpack8(const uint4& v, float (&f)[8])
{
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        f[2 * i] = __uint_as_float(w[i] << 16);
        f[2 * i + 1] = __uint_as_float(w[i] & 0xffff0000u);
    }
}
__device__ __forceinline__ uint4 pack8(const float (&f)[8])
{
    uint32_t h[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const __nv_bfloat162 p2 = __floats2bfloat162_rn(f[2 * i], f[2 * i + 1]);
        h[i] = *reinterpret_cast<const uint32_t*>(&p2);
    }
    return make_uint4(h[0], h[1], h[2], h[3]);
}

// ---------------------------------------------------------------------------------------
// Forward (and transposed) convolution on the 5th-generation tensor cores: an implicit GEMM
// with M = 128 voxels per block, N = the block's output channels (up to 256, one MMA wide),
// K = 27 taps x K input channels, flattened tap-major, in stages of 64 consecutive elements
// (four MMAs of K = 16; a stage spans several taps when K < 64). Operands sit in shared
// memory in the K-major layout with 128-byte swizzling:
// each 8-row group is one 1024-byte atom whose row r holds the stage's 64 elements as eight
// 16-byte chunks, chunk j stored at position j ^ (r mod 8); a descriptor with stride offset
// 1024 (next atom) whose start advances by 32 bytes per 16-channel slice describes any
// K = 16 slice. With this layout the eight lanes that copy one voxel row read its 128
// contiguous bytes and write eight distinct bank groups. The accumulators (FP32) live in
// tensor memory; one thread issues the MMAs. A ring of shared-memory stages is filled by
// asynchronous copies (cp.async, L1-cached, zero-filled outside the volume); the MMAs of a
// stage signal an mbarrier when they complete, which frees its buffer for the copies of a
// later stage. The epilogue reads the accumulators back with tcgen05.ld (warp w holds rows
// 32w..32w+31), adds the bias, applies the ReLU and stores. Every wait is bounded; a wait
// that gives up records it in g_sg_tc_fail (read by sg_check), and the block still releases
// its tensor memory.
// ---------------------------------------------------------------------------------------
constexpr int kTM = 128;         // voxels per block (MMA M)
constexpr int kTKC = 64;         // reduction elements per stage: one swizzle atom row (128 bytes)
#ifndef SG_TC_STAGES
#define SG_TC_STAGES 2
#endif
constexpr int kTStages = SG_TC_STAGES;  // shared-memory ring
constexpr int kTThreads = 128;   // four warps: one accumulator row per thread
constexpr int kTMaxN = 256;      // output channels per block (MMA N)
constexpr int kTAtom = 1024;     // one 8-row group: 8 rows x 128 bytes
constexpr int kTABytes = (kTM / 8) * kTAtom;
constexpr int kTPieces = kTM * 8 / kTThreads;  // 16-byte A pieces per thread and stage
constexpr long long kTWaitNs = 1000000000LL;  // a wait gives up after 1 s of the global timer

__device__ int g_sg_tc_fail;

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// byte offset of 16-byte chunk j of row r in a 128-byte-swizzled K-major tile
__device__ __forceinline__ uint32_t swz(int r, int j)
{
    return (uint32_t)((r >> 3) * kTAtom + (r & 7) * 128 + ((j ^ (r & 7)) << 4));
}

// shared-memory matrix descriptor: start address, stride byte offset 1024 (next 8-row atom),
// leading offset unused with swizzling (1), descriptor version 1 (bit 46), 128-byte
// swizzling (mode 2, bits 61-63)
__device__ __forceinline__ uint64_t tc_desc(uint32_t addr)
{
    return (uint64_t)((addr & 0x3FFFFu) >> 4) | (1ull << 16) | ((uint64_t)(kTAtom >> 4) << 32) | (1ull << 46) |
           (2ull << 61);
}

// instruction descriptor of kind::f16: FP32 accumulator, BF16 A and B, both K-major,
// N >> 3 at bit 17, M >> 4 at bit 24
__host__ __device__ constexpr uint32_t tc_idesc(int n)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(kTM >> 4) << 24);
}

// 16-byte asynchronous copy global -> shared (zero-filled beyond `bytes`), through L1, where
// the tap-shifted tiles of one block overlap
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, uint32_t bytes)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}

__device__ __forceinline__ unsigned long long tc_now_ns()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Wait for the phase of parity `parity` of an mbarrier to complete; false after kTWaitNs, or
// once `fail` (a flag in shared memory that another waiter set) is nonzero; the wait that runs
// out sets it. The global timer is read only every 64 polls: reading it costs hundreds of
// clocks, as much as the stage of a convolution.
__device__ __forceinline__ bool mbar_wait_or(uint32_t bar, uint32_t parity, volatile int* fail)
{
    unsigned long long t0 = 0;
    for (uint32_t poll = 1;; ++poll) {
        uint32_t done;
        asm volatile(
            "{\n.reg .pred q;\nmbarrier.try_wait.parity.shared::cta.b64 q, [%1], %2;\nselp.b32 %0, 1, 0, q;\n}"
            : "=r"(done)
            : "r"(bar), "r"(parity)
            : "memory");
        if (done) return true;
        if (fail && *fail) return false;
        if (poll % 64 == 0) {
            const unsigned long long t = tc_now_ns();
            if (t0 == 0) t0 = t;
            if ((long long)(t - t0) > kTWaitNs) {
                if (fail) *fail = 1;
                return false;
            }
        }
    }
}
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity) { return mbar_wait_or(bar, parity, nullptr); }

// one lane of a converged warp
__device__ __forceinline__ bool elect_one()
{
    uint32_t r;
    asm volatile("{\n.reg .pred p;\nelect.sync _|p, 0xffffffff;\nselp.b32 %0, 1, 0, p;\n}" : "=r"(r));
    return r != 0;
}

// Epilogue of the tensor-core convolutions: warp w reads accumulator rows 32w..32w+31 (its
// lanes' voxels) from tensor memory, adds the bias, applies the ReLU and stores BF16, FP32 and
// second outputs of voxel e of the batch (skipped when negative), channels n0..n0+BN-1.
__device__ __forceinline__ void conv_store_row(const ConvArgs& a, uint32_t tmem, int warp, long long e, int n0, int BN)
{
    for (int c0 = 0; c0 < BN; c0 += 16) {
        uint32_t r[16];
        const uint32_t addr = tmem + ((uint32_t)(32 * warp) << 16) + (uint32_t)c0;
        asm volatile(
            "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
            : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
              "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
            : "r"(addr));
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
        if (e >= 0) {
            const size_t o = (size_t)e * a.N + n0 + c0;
            float f[16];
#pragma unroll
            for (int c = 0; c < 16; ++c) {
                float t = __uint_as_float(r[c]) + (a.bias ? a.bias[n0 + c0 + c] : 0.0f);
                f[c] = a.relu ? fmaxf(t, 0.0f) : t;
            }
            if (a.y || a.y2) {
                uint4 h[2];
#pragma unroll
                for (int k = 0; k < 2; ++k) {
                    const float f8[8] = {f[8 * k],     f[8 * k + 1], f[8 * k + 2], f[8 * k + 3],
                                         f[8 * k + 4], f[8 * k + 5], f[8 * k + 6], f[8 * k + 7]};
                    h[k] = pack8(f8);
                }
                if (a.y) {
                    uint4* dst = reinterpret_cast<uint4*>(a.y + o);
                    dst[0] = h[0];
                    dst[1] = h[1];
                }
                if (a.y2) {
                    const uint4* src = reinterpret_cast<const uint4*>(a.other + o);
                    uint4* dst = reinterpret_cast<uint4*>(a.y2 + o);
#pragma unroll
                    for (int k = 0; k < 2; ++k) {
                        float g8[8], o8[8];
                        unpack8(h[k], g8);
                        unpack8(__ldg(src + k), o8);
#pragma unroll
                        for (int c = 0; c < 8; ++c) g8[c] = a.mode == kMask ? (o8[c] > 0.0f ? g8[c] : 0.0f) : g8[c] + o8[c];
                        dst[k] = pack8(g8);
                    }
                }
            }
            if (a.yf) {
                float4* dst = reinterpret_cast<float4*>(a.yf + o);
#pragma unroll
                for (int c = 0; c < 4; ++c) dst[c] = make_float4(f[4 * c], f[4 * c + 1], f[4 * c + 2], f[4 * c + 3]);
            }
        }
        __syncwarp();
    }
}

template <int kK>  // input channels, 0: a.K at run time
__global__ void __launch_bounds__(kTThreads) k_conv_tc(const ConvArgs a)
{
    extern __shared__ __align__(1024) unsigned char tc_smem_raw[];
    __shared__ __align__(8) uint64_t mbar[kTStages];
    __shared__ uint32_t tmem_base;
    const int tid = threadIdx.x, warp = tid >> 5;
    const int n0 = blockIdx.y * kTMaxN;
    const int BN = a.N - n0 < kTMaxN ? a.N - n0 : kTMaxN;  // a multiple of 16
    const int BBytes = (BN / 8) * kTAtom;
    // operand atoms must start on 1024-byte boundaries (the swizzle pattern is anchored there)
    unsigned char* tc_smem = tc_smem_raw + ((kTAtom - (smem_u32(tc_smem_raw) & (kTAtom - 1))) & (kTAtom - 1));
    unsigned char* sA = tc_smem;
    unsigned char* sB = tc_smem + kTStages * kTABytes;
    const int b = blockIdx.z;
    const int v = blockIdx.x * kTM + tid;  // this thread's result row
    // A pieces of this thread: piece p = tid + 128 i covers row p / 8, chunk p % 8 (the
    // chunk is the same for every i)
    const int pj = tid & 7;
    // source voxel of every (tap, row) of the block, periodic (-1: the row lies beyond the
    // volume), computed once: thread t fills row t
    __shared__ int s_src[27][kTM];
    {
        int x = 0, y = 0, z = 0;
        if (v < a.V) {
            x = v % a.W;
            y = (v / a.W) % a.H;
            z = v / (a.W * a.H);
        }
        for (int tap = 0; tap < 27; ++tap) {
            const int dz = tap / 9 - 1, dy = (tap / 3) % 3 - 1, dx = tap % 3 - 1;
            s_src[tap][tid] = v < a.V ? x_voxel(a.up, a.D, a.H, a.W, 0, wrap(z + a.sign * dz, a.D),
                                                wrap(y + a.sign * dy, a.H), wrap(x + a.sign * dx, a.W))
                                      : -1;
        }
    }
    // stages: 64 consecutive elements of the flattened (tap, channel) reduction index (tap
    // major); a 16-byte chunk never straddles two taps since K is a multiple of 16
    const int K = kK ? kK : a.K;
    const int nst = (27 * K + kTKC - 1) / kTKC;
    uint32_t ncols = 32;
    while ((int)ncols < BN) ncols <<= 1;
    if (tid == 0) {
        for (int s = 0; s < kTStages; ++s) asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&mbar[s])));
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base)),
                     "r"(ncols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = tmem_base;
    const bf16* xb = a.x + (size_t)b * (a.up ? a.V / 8 : a.V) * a.K;

    // reduction elements of stage st (a multiple of 16), and the tap and channel of chunk j
    auto stage_kc = [&](int st) { return 27 * K - st * kTKC < kTKC ? 27 * K - st * kTKC : kTKC; };
    auto chunk_of = [&](int st, int j, int& tap, int& ch) {
        const int e = st * kTKC + 8 * j;
        tap = e / K;
        ch = e - tap * K;
    };

    // asynchronous copies of stage st into ring buffer buf
    auto load_stage = [&](int st, int buf) {
        const int kc = stage_kc(st);
        const uint32_t abase = smem_u32(sA + buf * kTABytes);
        if (pj < kc / 8) {
            int tap, ch;
            chunk_of(st, pj, tap, ch);
#pragma unroll
            for (int i = 0; i < kTPieces; ++i) {
                const int row = (tid + kTThreads * i) >> 3;
                const int sv = s_src[tap][row];
                // any valid address (zero-filled) when the row lies outside the volume
                const bf16* src = xb + (sv >= 0 ? (size_t)sv * K + ch : 0);
                cp_async16(abase + swz(row, pj), src, sv >= 0 ? 16u : 0u);
            }
        }
        const uint32_t bbase = smem_u32(sB + buf * BBytes);
        for (int p = tid; p < BN * 8; p += kTThreads) {
            const int n = p >> 3, j = p & 7;
            if (j < kc / 8) {
                int tap, ch;
                chunk_of(st, j, tap, ch);
                cp_async16(bbase + swz(n, j), a.w + ((size_t)tap * a.N + n0 + n) * K + ch, 16u);
            }
        }
    };

    bool ok = true;
    for (int s = 0; s < kTStages - 1; ++s) {
        if (s < nst) load_stage(s, s);
        asm volatile("cp.async.commit_group;" ::: "memory");
    }
    for (int st = 0; st < nst; ++st) {
        const int buf = st % kTStages;
        // refill: stage st + kTStages - 1 goes to the buffer that stage st - 1's MMAs read
        const int nxt = st + kTStages - 1;
        if (nxt < nst) {
            if (st >= 1) ok = mbar_wait(smem_u32(&mbar[(st - 1) % kTStages]), (uint32_t)(((st - 1) / kTStages) & 1));
            if (ok) load_stage(nxt, nxt % kTStages);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
        asm volatile("cp.async.wait_group %0;" ::"n"(kTStages - 1) : "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        if (__syncthreads_or(!ok)) {
            ok = false;
            break;
        }
        if (tid == 0) {
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const int kc = stage_kc(st);
            const uint32_t abase = smem_u32(sA + buf * kTABytes), bbase = smem_u32(sB + buf * BBytes);
            const uint32_t idesc = tc_idesc(BN);
            for (int kk = 0; kk < kc; kk += 16) {
                const uint64_t ad = tc_desc(abase + kk * 2), bd = tc_desc(bbase + kk * 2);
                const uint32_t accum = (st > 0 || kk > 0) ? 1u : 0u;
                asm volatile(
                    "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
                    "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(tmem),
                    "l"(ad), "l"(bd), "r"(idesc), "r"(accum));
            }
            asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                             smem_u32(&mbar[buf]))
                         : "memory");
        }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    // the last stage's commit covers every MMA of the block (they complete in order)
    if (ok) ok = mbar_wait(smem_u32(&mbar[(nst - 1) % kTStages]), (uint32_t)(((nst - 1) / kTStages) & 1));
    if (!ok && tid == 0) atomicExch(&g_sg_tc_fail, 1);
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (__syncthreads_and(ok)) conv_store_row(a, tmem, warp, v < a.V ? (long long)b * a.V + v : -1, n0, BN);
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(ncols));
}

// ---------------------------------------------------------------------------------------
// The same convolution marching along y (W >= 3, K = 16, 32, 64, 96 or 128): the kernel of the
// network's layers. Measured, forward on one box (tap by tap -> marching): 128^3,
// 32 -> 32 channels 463 -> 167 us, 64 -> 32 643 -> 238 us; 64^3, 64 -> 64 171 -> 60 us (960
// TFLOP/s); 32^3, 96 -> 96 60 -> 29 us; 16^3, 128 -> 128 59 -> 15 us.
//
// What bounds a tap-by-tap implicit GEMM with few output channels is shared memory: every
// K = 16 slice of every tap reads the 128 x 16 operand A (4 KB, 32 clocks) for as little as
// 16 clocks of products (N = 32), and every tap's rows are copied in again. Here a block
// computes T consecutive rows (y) of one column of 128 voxels and takes each source row once
// per dz:
//  * the three taps dy that read one source row go to three neighbouring output rows, whose
//    accumulators are neighbouring column ranges of tensor memory: one MMA with the three taps'
//    weights side by side (N' = 3 N columns) serves all three (two or one at the ends of the
//    strip), so operand A is read a third as often;
//  * the taps dx read the same staged row through descriptors that start one row earlier or
//    later (the 128-byte swizzle is keyed to the absolute shared-memory address), so a row is
//    copied 3 (T + 2) / T times instead of 27.
// The column of 128 voxels is any 16 groups of 8 x-neighbours (b, z, x / 8): each group is
// staged as 10 rows of 128 bytes, its voxels with their left and right neighbour (periodic),
// and the descriptor's stride between 8-row groups is 1280 bytes. So a box of any W that is a
// multiple of 8 fills the MMA's 128 rows (other widths end each row with a short group).
// Per accumulator the products are added in the order of k_conv_tc (taps ascending, then
// channels): source rows ascend for sign = +1 and descend for sign = -1, and outputs are
// bitwise the same.
// A persistent block of 14 warps: 4 epilogue warps (tensor memory -> bias, ReLU -> global,
// one accumulator set while the other is being computed), one warp that issues the MMAs, one
// that loads weights (TMA; one dz at a time in two buffers, or all of them once per block where
// they fit), 8 warps that copy rows (cp.async: a TMA box can't wrap around) into a ring of up
// to eight. The copies of a thread are the same pieces of every row, so that one costs an
// address and a copy instruction: with four warps and the addresses formed per piece the
// copying warps were the limit at 1000 clocks a row.
// Every wait is bounded; one that gives up sets a flag in shared memory that ends every role
// and is reported through g_sg_tc_fail.
// ---------------------------------------------------------------------------------------
constexpr int kMCopy = 256;              // copying threads
constexpr int kMThreads = 192 + kMCopy;
constexpr int kMRows = kColumnRows;      // staged rows: 16 groups of 8 voxels with two neighbours
constexpr int kMChunk = kMRows * 128;  // bytes of 64 channels of a staged row
constexpr int kMStages = 8;      // most ring stages
constexpr int kMSmem = kBlockSmem;

struct MarchArgs {
    ConvArgs c;
    int GX, NG;           // groups per x-row, groups over the batch
    int T, nstrip;        // output rows per unit, strips along y
    int NB, nblk;         // output channels per unit, channel blocks
    int units;            // columns x strips x channel blocks
    int nA;               // ring stages
    int resident;         // all weights loaded once per block (nblk = 1)
    int bufs;             // accumulator sets
    uint32_t ncols;       // tensor-memory columns
};

// barrier 1 over the copying threads, true when `v` is true in all of them
__device__ __forceinline__ bool bar_and(bool v)
{
    uint32_t r;
    asm volatile(
        "{\n.reg .pred p, q;\nsetp.ne.b32 p, %1, 0;\nbarrier.cta.red.and.pred q, 1, %2, p;\nselp.b32 %0, 1, 0, q;\n}"
        : "=r"(r)
        : "r"((uint32_t)v), "n"(kMCopy)
        : "memory");
    return r != 0;
}

__device__ __forceinline__ void mbar_arrive(uint32_t bar)
{
    asm volatile("{\n.reg .b64 t;\nmbarrier.arrive.shared::cta.b64 t, [%0];\n}" ::"r"(bar) : "memory");
}

__device__ __forceinline__ void tc_commit(uint32_t bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

__device__ __forceinline__ void tc_mma(uint32_t d, uint64_t ad, uint64_t bd, uint32_t idesc, uint32_t accum)
{
    asm volatile(
        "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(d),
        "l"(ad), "l"(bd), "r"(idesc), "r"(accum)
        : "memory");
}

// K-major 128-byte-swizzled descriptor with `stride` bytes between 8-row groups (tc_desc: 1024)
__device__ __forceinline__ uint64_t tc_desc_stride(uint32_t addr, uint32_t stride)
{
    return (uint64_t)((addr & 0x3FFFFu) >> 4) | (1ull << 16) | ((uint64_t)(stride >> 4) << 32) | (1ull << 46) |
           (2ull << 61);
}

template <int kK>
__global__ void __launch_bounds__(kMThreads, 1) k_conv_march(const __grid_constant__ MarchArgs m, const __grid_constant__ CUtensorMap wmap)
{
    constexpr int kCh = (kK + 63) / 64;   // 64-channel chunks of a staged row
    constexpr int kKC = kK / 8;           // 16-byte pieces of a voxel
    constexpr uint32_t kABytes = kCh * kMChunk;
    extern __shared__ __align__(1024) unsigned char tc_smem_raw[];
    __shared__ __align__(8) uint64_t s_full[kMStages], s_empty[kMStages], s_bfull[3], s_bempty[2], s_afull[2],
        s_aempty[2], s_drain;
    __shared__ uint32_t s_tmem;
    __shared__ int s_fail;
    __shared__ int s_off[kMRows];  // source voxel of each staged row at y = 0 (-1: no such voxel)
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t base = (smem_u32(tc_smem_raw) + kTAtom - 1) & ~(uint32_t)(kTAtom - 1);
    const int NB = m.NB;
    const uint32_t btap = (uint32_t)(3 * NB) * 128u;   // weights of one (dz, dx), one chunk: rows (dy block, n)
    const uint32_t bbytes = 3u * kCh * btap;           // weights of one dz
    const uint32_t sA = base + (m.resident ? 3u : 2u) * bbytes;
    if (tid == 0) {
        for (int s = 0; s < kMStages; ++s) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(&s_full[s])), "n"(kMCopy));
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&s_empty[s])));
        }
        for (int s = 0; s < 3; ++s) asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&s_bfull[s])));
        for (int s = 0; s < 2; ++s) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&s_bempty[s])));
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&s_afull[s])));
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 4;" ::"r"(smem_u32(&s_aempty[s])));
        }
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&s_drain)));
        s_fail = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)),
                     "r"(m.ncols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = s_tmem;
    volatile int* fail = &s_fail;
    const int H = m.c.H, W = m.c.W, sign = m.c.sign;
    const int step = (int)gridDim.x;

    if (warp >= 6) {
        // ---- copies of source rows ----
        constexpr int kP = (kMRows * kKC + kMCopy - 1) / kMCopy;  // 16-byte pieces per thread and row
        const int pt = tid - 192;
        int slot = 0;        // ring slot of the next stage
        uint32_t round = 0;  // times the ring has been filled before
        bool ok = true, all = true;  // all: no copying thread has given up (the same in every one of them)
        for (int u = blockIdx.x; u < m.units && all; u += step) {
            const int q = u / m.nblk;
            const int strip = q % m.nstrip, tc = q / m.nstrip;
            const int y0 = strip * m.T, te = min(m.T, H - y0);
            for (int d = 0; d < 3; ++d) {
                // the table's last readers are done; leave together when one of them gave up
                all = bar_and(ok);
                if (!all) break;
                for (int row = pt; row < kMRows; row += kMCopy) {
                    const int g = tc * 16 + row / 10;
                    int off = -1;
                    if (g < m.NG) {
                        const int xg = g % m.GX, r = g / m.GX;
                        const int z = r % m.c.D, b = r / m.c.D;
                        const int x = 8 * xg - 1 + row % 10;  // beyond W: past the row's last neighbour
                        if (x <= W) off = x_voxel(m.c.up, m.c.D, H, W, b, wrap(z + sign * (d - 1), m.c.D), 0, wrap(x, W));
                    }
                    s_off[row] = off;
                }
                asm volatile("barrier.cta.sync 1, %0;" ::"n"(kMCopy) : "memory");
                int voff[kP];  // source voxel (at y = 0) of this thread's pieces of a row
#pragma unroll
                for (int i = 0; i < kP; ++i) {
                    const int p = pt + kMCopy * i;
                    voff[i] = p < kMRows * kKC ? s_off[p / kKC] : -1;
                }
                for (int rr = 0; rr < te + 2; ++rr) {
                    const int ys = wrap(y0 - 1 + (sign > 0 ? rr : te + 1 - rr), H);
                    if (round > 0) ok = mbar_wait_or(smem_u32(&s_empty[slot]), (round - 1) & 1u, fail);
                    if (!ok) break;
                    const uint32_t dst = sA + (uint32_t)slot * kABytes;
                    const bf16* xr = m.c.x + (size_t)(m.c.up ? (ys >> 1) * (W >> 1) : ys * W) * kK;
#pragma unroll
                    for (int i = 0; i < kP; ++i) {
                        const int p = pt + kMCopy * i, row = p / kKC, j = p - row * kKC;
                        if (voff[i] >= 0)
                            cp_async16(dst + (uint32_t)((j >> 3) * kMChunk + row * 128 + (((j & 7) ^ (row & 7)) << 4)),
                                       xr + (size_t)voff[i] * kK + 8 * j, 16u);
                    }
                    // this thread's arrival at the stage's barrier, once its copies have landed
                    asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(smem_u32(&s_full[slot]))
                                 : "memory");
                    if (++slot == m.nA) {
                        slot = 0;
                        ++round;
                    }
                }
            }
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
    } else if (warp == 5) {
        // ---- weights: those of one dz as nine boxes (dx, dy) of NB rows and 64 channels ----
        if (lane == 0) {
            int loads = 0;
            bool ok = true;
            for (int u = blockIdx.x; u < m.units && ok; u += step) {
                const int n0 = (u % m.nblk) * NB;
                if (m.resident && loads > 0) break;
                for (int d = 0; d < 3; ++d, ++loads) {
                    const int b = m.resident ? d : loads & 1;
                    if (!m.resident && loads >= 2)
                        ok = mbar_wait_or(smem_u32(&s_bempty[b]), (uint32_t)((loads >> 1) - 1) & 1u, fail);
                    if (!ok) break;
                    const uint32_t bar = smem_u32(&s_bfull[b]);
                    asm volatile("{\n.reg .b64 t;\nmbarrier.arrive.expect_tx.shared::cta.b64 t, [%0], %1;\n}" ::"r"(bar),
                                 "r"(bbytes)
                                 : "memory");
                    for (int dx = 0; dx < 3; ++dx)
                        for (int ch = 0; ch < kCh; ++ch)
                            for (int blk = 0; blk < 3; ++blk) {
                                const int tap = 9 * d + 3 * (sign * (1 - blk) + 1) + dx;
                                asm volatile(
                                    "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes "
                                    "[%0], [%1, {%3, %4, %5}], [%2];" ::"r"(base + (uint32_t)b * bbytes +
                                                                            (uint32_t)(dx * kCh + ch) * btap +
                                                                            (uint32_t)(blk * NB) * 128u),
                                    "l"(&wmap), "r"(bar), "r"(64 * ch), "r"(n0), "r"(tap)
                                    : "memory");
                            }
                }
            }
            // no load may be in flight when the block ends (also after a failure elsewhere)
            for (int k = max(0, loads - (m.resident ? 3 : 2)); k < loads; ++k)
                mbar_wait(smem_u32(&s_bfull[m.resident ? k : k & 1]), m.resident ? 0u : (uint32_t)(k >> 1) & 1u);
        }
        __syncwarp();
    } else if (warp == 4) {
        // ---- MMAs: the warp stays converged (so that addresses stay in uniform registers) and
        // one elected lane issues ----
        const bool lead = elect_one();
        int slot = 0, nu = 0;
        uint32_t round = 0;
        int nb_used = 0;
        bool ok = true;
        const int jfirst = sign > 0 ? 2 : 0;  // the block of the tap dy = -1: its output row's first
        for (int u = blockIdx.x; u < m.units && ok; u += step, ++nu) {
            const int strip = (u / m.nblk) % m.nstrip;
            const int te = min(m.T, H - strip * m.T);
            const int buf = m.bufs == 2 ? nu & 1 : 0;
            const uint32_t acc = tmem + (uint32_t)(buf * m.T * NB);
            const int use = m.bufs == 2 ? nu >> 1 : nu;
            if (use > 0) ok = mbar_wait_or(smem_u32(&s_aempty[buf]), (uint32_t)(use - 1) & 1u, fail);
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            for (int d = 0; d < 3 && ok; ++d) {
                const int bb = m.resident ? d : nb_used & 1;
                const uint32_t sB = base + (uint32_t)bb * bbytes;
                if (!m.resident || nb_used < 3) {
                    ok = mbar_wait_or(smem_u32(&s_bfull[bb]), m.resident ? 0u : (uint32_t)(nb_used >> 1) & 1u, fail);
                    ok = __all_sync(0xffffffffu, ok);
                    if (!ok) break;
                }
                for (int rr = 0; rr < te + 2; ++rr) {
                    const int r = sign > 0 ? rr : te + 1 - rr;
                    ok = mbar_wait_or(smem_u32(&s_full[slot]), round & 1u, fail);
                    ok = __all_sync(0xffffffffu, ok);
                    if (!ok) break;
                    // the copies' writes, ordered before this thread by the barrier, are made
                    // visible to the tensor core's reads (here and not in the copying
                    // threads, where the fence would wait for every copy in flight)
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    const int jlo = max(0, 2 - r), jhi = min(2, te + 1 - r);
                    const uint32_t dcol = acc + (uint32_t)((r - 2 + jlo) * NB);
                    const uint32_t idesc = tc_idesc((jhi - jlo + 1) * NB);
                    const uint64_t a0 = tc_desc_stride(sA + (uint32_t)slot * kABytes + 128u, 1280u);
                    const uint64_t b0 = tc_desc_stride(sB + (uint32_t)(jlo * NB) * 128u, kTAtom);
                    if (lead) {
#pragma unroll
                        for (int dx = 0; dx < 3; ++dx) {
#pragma unroll
                            for (int sl = 0; sl < kK / 16; ++sl) {
                                // descriptor addresses count 16 bytes
                                const uint64_t ad = a0 + (uint64_t)((sl >> 2) * (kMChunk / 16) + (sl & 3) * 2) +
                                                    (uint64_t)(int64_t)(sign * (dx - 1) * 8);
                                const uint64_t bd = b0 + (uint64_t)((uint32_t)(dx * kCh + (sl >> 2)) * (btap / 16u)) +
                                                    (uint64_t)((sl & 3) * 2);
                                if (dx == 0 && sl == 0 && d == 0 && jfirst >= jlo && jfirst <= jhi) {
                                    // this row is the first of output row r - 2 + jfirst: its
                                    // accumulator starts here, the others go on
                                    const uint32_t fo = (uint32_t)((jfirst - jlo) * NB);
                                    tc_mma(dcol + fo, ad, bd + fo * 8u, tc_idesc(NB), 0u);
                                    if (jhi > jlo) {
                                        const uint32_t ro = jfirst == jlo ? (uint32_t)NB : 0u;
                                        tc_mma(dcol + ro, ad, bd + ro * 8u, tc_idesc((jhi - jlo) * NB), 1u);
                                    }
                                } else {
                                    tc_mma(dcol, ad, bd, idesc, 1u);
                                }
                            }
                        }
                        tc_commit(smem_u32(&s_empty[slot]));
                    }
                    if (++slot == m.nA) {
                        slot = 0;
                        ++round;
                    }
                }
                if (ok && !m.resident && lead) tc_commit(smem_u32(&s_bempty[nb_used & 1]));
                ++nb_used;
            }
            if (ok && lead) tc_commit(smem_u32(&s_afull[buf]));
        }
        if (!ok && lead) {
            // MMAs issued before the failure still use this block's memories: wait for them
            tc_commit(smem_u32(&s_drain));
            mbar_wait(smem_u32(&s_drain), 0u);
        }
        __syncwarp();
    } else {
        // ---- epilogue ----
        int nu = 0;
        bool ok = true;
        for (int u = blockIdx.x; u < m.units; u += step, ++nu) {
            const int nbk = u % m.nblk, q = u / m.nblk;
            const int strip = q % m.nstrip, tc = q / m.nstrip;
            const int y0 = strip * m.T, te = min(m.T, H - y0);
            const int buf = m.bufs == 2 ? nu & 1 : 0;
            const int use = m.bufs == 2 ? nu >> 1 : nu;
            const int g = tc * 16 + tid / 8;
            const int xg = g % m.GX, r = g / m.GX;   // r = b D + z
            const int x = 8 * xg + (tid & 7);
            const long long v0 = g < m.NG && x < W ? ((long long)r * H + y0) * W + x : -1;
            ok = mbar_wait_or(smem_u32(&s_afull[buf]), (uint32_t)use & 1u, fail);
            if (!__all_sync(0xffffffffu, ok)) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            for (int t = 0; t < te; ++t)
                conv_store_row(m.c, tmem + (uint32_t)((buf * m.T + t) * NB), warp, v0 < 0 ? -1 : v0 + (long long)t * W,
                               nbk * NB, NB);
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&s_aempty[buf]));
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (tid == 0 && s_fail) atomicExch(&g_sg_tc_fail, 1);
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(m.ncols));
}

// ---------------------------------------------------------------------------------------
// Weight gradient on the 5th-generation tensor cores (W >= 3): dW[tap][ci][co] is a
// product over voxels of x rows and dy rows, both channels-last, i.e. both operands with the
// reduction index (voxels) as rows of shared memory: MN-major operands. What bounds a
// tap-by-tap kernel is reading x and dy once per tap (27 times); here a unit takes one dz, a
// block of CI input and CO output channels, a column of 128 voxels (16 groups of 8
// x-neighbours, as in k_conv_march) and T rows of x:
//  * N = 3 CI: the three taps dx are three column blocks of one operand, the staged x row
//    read from row 0, 1 and 2 of each 10-row group: the descriptor's stride between
//    64-, 32- or 16-channel blocks is one staged row;
//  * M = 3 CO (padded to 128, or two tiles of 128 for CO = 64): the three taps dy are the dy
//    rows y + 1, y, y - 1, neighbouring slots of a ring: the stride between channel blocks is
//    one slot. The ring's first two slots are copied a second time behind its end, so that
//    three consecutive rows are always consecutive slots; rows of M beyond 3 CO read whatever
//    the next slots hold and are dropped.
// A copy waits until both the x slot and the dy slots that it overwrites have been read
// (WgradUnits in wgrad_plan.cuh, with the plan).
// So x and dy are read three times in all (once per dz), and an MMA of K = 16 voxels serves
// nine taps. Rows of 128, 64 or 32 bytes use the swizzle of that width. A unit's sums (T rows,
// at most 2048 voxels: partial sums stay as short as those of the kernel below) are added to
// dw with one reduction per element, 32 consecutive output channels per warp.
// Measured (tap by tap with mma.sync -> this): one 128^3 box 32 -> 32 channels 2266 -> 157 us,
// 64 -> 32 2297 -> 208 us (1117 TFLOP/s); 64^3 64 -> 64 365 -> 60 us; 16^3 128 -> 128 56 -> 13 us.
// 13 warps: 4 epilogue, 1 MMA, 8 copies (cp.async, zero-filled beyond the row or batch).
// Waits are bounded as in k_conv_march.
// ---------------------------------------------------------------------------------------
constexpr int kGThreads = 160 + kMCopy;

struct WgradTcArgs {
    const bf16* x;
    const bf16* dy;
    float* dw;
    int D, H, W, Cin, Cout;
    int up;              // x is the coarse grid, read as its nearest upsampling
    WgradPlan p;
};

// MN-major descriptor: `lbo` bytes between channel blocks of one swizzle width, `sbo` between
// groups of 8 rows; swizzle mode of a row of `row` bytes
template <int kRow>
__device__ __forceinline__ uint64_t tc_desc_mn(uint32_t addr, uint32_t lbo, uint32_t sbo)
{
    constexpr uint64_t mode = kRow == 128 ? 2 : (kRow == 64 ? 4 : 6);
    return (uint64_t)((addr & 0x3FFFFu) >> 4) | ((uint64_t)(lbo >> 4) << 16) | ((uint64_t)(sbo >> 4) << 32) |
           (1ull << 46) | (mode << 61);
}

// offset of 16-byte piece j of a row of kRow bytes under that swizzle (slots start on 1024 bytes)
template <int kRow>
__device__ __forceinline__ uint32_t swz_row(int r, int j)
{
    return (uint32_t)(r * kRow + ((j ^ (((r * kRow) >> 7) & (kRow / 16 - 1))) << 4));
}

template <int kCI, int kCO>
__global__ void __launch_bounds__(kGThreads, 1) k_wgrad_tc(const __grid_constant__ WgradTcArgs m)
{
    constexpr int kRX = 2 * kCI, kRY = 2 * kCO;              // bytes of a staged row
    constexpr uint32_t kXB = kMRows * kRX, kYB = kTM * kRY;  // bytes of a slot
    constexpr int kTiles = kCO == 64 ? 2 : 1, kN = 3 * kCI;
    extern __shared__ __align__(1024) unsigned char tc_smem_raw[];
    __shared__ __align__(8) uint64_t s_full[kGStages], s_empty[kGStages], s_afull[2], s_aempty[2], s_drain;
    __shared__ uint32_t s_tmem;
    __shared__ int s_fail;
    __shared__ int s_xoff[kMRows], s_yoff[kTM];  // voxels of the staged rows at y = 0 (-1: none)
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t base = (smem_u32(tc_smem_raw) + kTAtom - 1) & ~(uint32_t)(kTAtom - 1);
    const int R = m.p.slots();
    const uint32_t sX = base, sY = base + (uint32_t)m.p.nX * kXB;
    if (tid == 0) {
        for (int s = 0; s < kGStages; ++s) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(&s_full[s])), "n"(kMCopy));
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&s_empty[s])));
        }
        for (int s = 0; s < 2; ++s) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&s_afull[s])));
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 4;" ::"r"(smem_u32(&s_aempty[s])));
        }
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&s_drain)));
        s_fail = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)),
                     "r"(m.p.ncols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = s_tmem;
    volatile int* fail = &s_fail;
    const int H = m.H, W = m.W, step = (int)gridDim.x;
    const int combos = m.p.combos();

    if (warp >= 5) {
        // ---- copies ----
        constexpr int kPX = kRX / 16, kPY = kRY / 16;
        constexpr int kNX = (kMRows * kPX + kMCopy - 1) / kMCopy, kNY = kTM * kPY / kMCopy;
        const int pt = tid - 160;
        int slot = 0, ys = 0;  // x slot of the next stage, dy slot of the next dy row
        uint32_t round = 0;
        int stage = 0;  // the next stage, over all units
        WgradUnits units;
        bool ok = true, all = true;
        for (int u = blockIdx.x; u < m.p.units && all; u += step) {
            const int combo = u % combos, q = u / combos;
            const int d = combo % 3, ci0 = (combo / 3) % m.p.nci * kCI, co0 = combo / (3 * m.p.nci) * kCO;
            const int strip = q % m.p.nstrip, tc = q / m.p.nstrip;
            const int y0 = strip * m.p.T, te = m.p.rows(u);
            all = bar_and(ok);
            if (!all) break;
            for (int row = pt; row < kMRows + kTM; row += kMCopy) {
                const bool isx = row < kMRows;
                const int r = isx ? row : row - kMRows;
                const int g = tc * 16 + (isx ? r / 10 : r / 8);
                int off = -1;
                if (g < m.p.NG) {
                    const int xg = g % m.p.GX, l = g / m.p.GX;
                    const int z = l % m.D, b = l / m.D;
                    const int x = isx ? 8 * xg - 1 + r % 10 : 8 * xg + r % 8;
                    if (isx && x <= W) off = x_voxel(m.up, m.D, H, W, b, wrap(z + d - 1, m.D), 0, wrap(x, W));
                    if (!isx && x < W) off = ((b * m.D + z) * H) * W + x;
                }
                if (isx)
                    s_xoff[r] = off;
                else
                    s_yoff[r] = off;
            }
            asm volatile("barrier.cta.sync 1, %0;" ::"n"(kMCopy) : "memory");
            int xo[kNX], yo[kNY];
#pragma unroll
            for (int i = 0; i < kNX; ++i) {
                const int p = pt + kMCopy * i;
                xo[i] = p < kMRows * kPX ? s_xoff[p / kPX] : -2;
            }
#pragma unroll
            for (int i = 0; i < kNY; ++i) yo[i] = s_yoff[(pt + kMCopy * i) / kPY];
            // dy row y into the next slot of the ring (and its copy behind the ring's end)
            auto load_y = [&](int y) {
                const bf16* src = m.dy + (size_t)y * W * m.Cout + co0;
#pragma unroll
                for (int i = 0; i < kNY; ++i) {
                    const int p = pt + kMCopy * i, row = p / kPY, j = p - row * kPY;
                    const bf16* s = src + (yo[i] >= 0 ? (size_t)yo[i] * m.Cout + 8 * j : 0);
                    const uint32_t at = sY + swz_row<kRY>(row, j), n = yo[i] >= 0 ? 16u : 0u;
                    cp_async16(at + (uint32_t)ys * kYB, s, n);
                    if (ys < 2) cp_async16(at + (uint32_t)(ys + R) * kYB, s, n);
                }
                ys = ys + 1 == R ? 0 : ys + 1;
            };
            const int w = units.first_waits_for(m.p, stage);
            if (w >= 0) ok = mbar_wait_or(smem_u32(&s_empty[w % m.p.nX]), (uint32_t)(w / m.p.nX) & 1u, fail);
            for (int i = 0; i < te; ++i) {
                if (ok && round > 0) ok = mbar_wait_or(smem_u32(&s_empty[slot]), (round - 1) & 1u, fail);
                if (!ok) break;
                if (i == 0) {
                    load_y(wrap(y0 - 1, H));
                    load_y(y0);
                }
                load_y(wrap(y0 + i + 1, H));
                const bf16* src = m.x + (size_t)(m.up ? ((y0 + i) >> 1) * (W >> 1) : (y0 + i) * W) * m.Cin + ci0;
#pragma unroll
                for (int k = 0; k < kNX; ++k) {
                    const int p = pt + kMCopy * k, row = p / kPX, j = p - row * kPX;
                    if (xo[k] != -2)
                        cp_async16(sX + (uint32_t)slot * kXB + swz_row<kRX>(row, j),
                                   src + (xo[k] >= 0 ? (size_t)xo[k] * m.Cin + 8 * j : 0), xo[k] >= 0 ? 16u : 0u);
                }
                asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(smem_u32(&s_full[slot]))
                             : "memory");
                if (++slot == m.p.nX) {
                    slot = 0;
                    ++round;
                }
            }
            stage += te;
            units.ended(stage);
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
    } else if (warp == 4) {
        // ---- MMAs ----
        constexpr uint32_t kIdesc = tc_idesc(kN) | (1u << 15) | (1u << 16);  // both operands MN-major
        const bool lead = elect_one();
        int slot = 0, ys = 0, nu = 0;
        uint32_t round = 0;
        bool ok = true;
        for (int u = blockIdx.x; u < m.p.units && ok; u += step, ++nu) {
            const int te = m.p.rows(u);
            const int buf = m.p.bufs == 2 ? nu & 1 : 0;
            const int use = m.p.bufs == 2 ? nu >> 1 : nu;
            const uint32_t acc = tmem + (uint32_t)(buf * kTiles * kN);
            if (use > 0) ok = mbar_wait_or(smem_u32(&s_aempty[buf]), (uint32_t)(use - 1) & 1u, fail);
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            for (int i = 0; i < te; ++i) {
                ok = mbar_wait_or(smem_u32(&s_full[slot]), round & 1u, fail);
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) break;
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint64_t a0 = tc_desc_mn<kRY>(sY + (uint32_t)ys * kYB, kYB, 8u * kRY);
                const uint64_t b0 = tc_desc_mn<kRX>(sX + (uint32_t)slot * kXB, kRX, 10u * kRX);
                if (lead) {
#pragma unroll
                    for (int k = 0; k < 8; ++k)
#pragma unroll
                        for (int t = 0; t < kTiles; ++t)
                            tc_mma(acc + (uint32_t)(t * kN), a0 + (uint64_t)(k * (16 * kRY / 16) + t * (2 * (int)kYB / 16)),
                                   b0 + (uint64_t)(k * (20 * kRX / 16)), kIdesc, (i > 0 || k > 0) ? 1u : 0u);
                    tc_commit(smem_u32(&s_empty[slot]));
                }
                ys = ys + 1 == R ? 0 : ys + 1;
                if (++slot == m.p.nX) {
                    slot = 0;
                    ++round;
                }
            }
            ys = ys + 2 >= R ? ys + 2 - R : ys + 2;  // the unit's last two dy rows
            if (ok && lead) tc_commit(smem_u32(&s_afull[buf]));
        }
        if (!ok && lead) {
            // MMAs issued before the failure still use this block's memories: wait for them
            tc_commit(smem_u32(&s_drain));
            mbar_wait(smem_u32(&s_drain), 0u);
        }
        __syncwarp();
    } else {
        // ---- epilogue: accumulator row = (dy block, output channel), column = (dx, input channel) ----
        int nu = 0;
        for (int u = blockIdx.x; u < m.p.units; u += step, ++nu) {
            const int combo = u % combos;
            const int d = combo % 3, ci0 = (combo / 3) % m.p.nci * kCI, co0 = combo / (3 * m.p.nci) * kCO;
            const int buf = m.p.bufs == 2 ? nu & 1 : 0;
            const int use = m.p.bufs == 2 ? nu >> 1 : nu;
            const bool ok = mbar_wait_or(smem_u32(&s_afull[buf]), (uint32_t)use & 1u, fail);
            if (!__all_sync(0xffffffffu, ok)) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
            for (int t = 0; t < kTiles; ++t) {
                if (t * 128 + 32 * warp >= 3 * kCO) continue;  // the whole warp's rows are padding
                const int r = t * 128 + tid, j = r / kCO;  // j > 2: padding
                // block j: dy row y - 1 + j, tap dy = 1 - j
                float* out = m.dw + ((size_t)(9 * d + 3 * (2 - min(j, 2))) * m.Cin + ci0) * m.Cout + co0 + (r - j * kCO);
#pragma unroll 1
                for (int c0 = 0; c0 < kN; c0 += 16) {
                    uint32_t v[16];
                    const uint32_t addr =
                        tmem + ((uint32_t)(32 * warp) << 16) + (uint32_t)((buf * kTiles + t) * kN + c0);
                    asm volatile(
                        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
                        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
                        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]),
                          "=r"(v[7]), "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]),
                          "=r"(v[14]), "=r"(v[15])
                        : "r"(addr));
                    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                    if (j < 3) {
                        float* o = out + ((size_t)(c0 / kCI) * m.Cin + c0 % kCI) * m.Cout;
#pragma unroll
                        for (int c = 0; c < 16; ++c) atomicAdd(o + (size_t)c * m.Cout, __uint_as_float(v[c]));
                    }
                    __syncwarp();
                }
            }
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&s_aempty[buf]));
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (tid == 0 && s_fail) atomicExch(&g_sg_tc_fail, 1);
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(m.p.ncols));
}

struct WgradArgs {
    const bf16* x;
    const bf16* dy;
    float* dw;
    int D, H, W, V, Cin, Cout;
    long long total;  // B * V voxels of the reduction
    int chunk;        // voxels per block (a multiple of 32)
    int ci_tiles;     // tiles of 64 input channels
    int up;           // x is the coarse grid, read as its nearest upsampling
};

// four 8x8 BF16 matrices from shared memory, transposed on the way (lanes 8j..8j+7 give the
// row addresses of matrix j): each lane receives (M[2(l%4)][l/4], M[2(l%4)+1][l/4]) of every
// matrix, which is the m16n8k16 fragment layout for an operand stored K-major
__device__ __forceinline__ void ldsm_x4_t(uint32_t& r0, uint32_t& r1, uint32_t& r2, uint32_t& r3, const bf16* p)
{
    const uint32_t addr = (uint32_t)__cvta_generic_to_shared(p);
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
                 : "r"(addr));
}

constexpr int kWM = 64, kWN = 64, kWS = 32, kWLd = 72, kWThreads = 128;

// Weight gradient of one tap (blockIdx.x % 27) over one chunk of voxels (blockIdx.x / 27) for
// one 64 x 64 tile of (input, output) channels (blockIdx.y): rows = input channels, columns =
// output channels, reduction over voxels in stages of 32. Both operands stay channels-last in
// shared memory ([voxel][channel], 144-byte rows) and the fragments come from transposing
// loads. The next stage is fetched into registers during the current one's products.
__global__ void __launch_bounds__(kWThreads) k_wgrad(const WgradArgs a)
{
    __shared__ __align__(16) bf16 Xs[2][kWS][kWLd];
    __shared__ __align__(16) bf16 Gs[2][kWS][kWLd];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int tap = blockIdx.x % 27;
    const long long e0 = (long long)(blockIdx.x / 27) * a.chunk;
    const long long e1 = e0 + a.chunk < a.total ? e0 + a.chunk : a.total;
    const int ci0 = (blockIdx.y % a.ci_tiles) * kWM, co0 = (blockIdx.y / a.ci_tiles) * kWN;
    const int dz = tap / 9 - 1, dy = (tap / 3) % 3 - 1, dx = tap % 3 - 1;
    const int lr = tid >> 2, lc = (tid & 3) * 16;  // this thread stages voxel row lr, 16 channels from lc
    const int ncols = a.Cout - co0 < kWN ? a.Cout - co0 : kWN;
    uint4 rx0, rx1, rg0, rg1;
    auto fetch = [&](long long e) {
        rx0 = rx1 = rg0 = rg1 = make_uint4(0u, 0u, 0u, 0u);
        const long long ev = e + lr;
        if (ev < e1) {
            const long long bb = ev / a.V;
            const int v = (int)(ev - bb * a.V);
            const int xa = v % a.W, ya = (v / a.W) % a.H, za = v / (a.W * a.H);
            const int xs = wrap(xa + dx, a.W), ys = wrap(ya + dy, a.H), zs = wrap(za + dz, a.D);
            const size_t src = (size_t)bb * (a.up ? a.V / 8 : a.V) + (size_t)x_voxel(a.up, a.D, a.H, a.W, 0, zs, ys, xs);
            if (ci0 + lc < a.Cin) {
                const bf16* p = a.x + src * a.Cin + ci0 + lc;
                rx0 = *reinterpret_cast<const uint4*>(p);
                rx1 = *reinterpret_cast<const uint4*>(p + 8);
            }
            if (co0 + lc < a.Cout) {
                const bf16* p = a.dy + (size_t)ev * a.Cout + co0 + lc;
                rg0 = *reinterpret_cast<const uint4*>(p);
                rg1 = *reinterpret_cast<const uint4*>(p + 8);
            }
        }
    };
    auto stash = [&](int buf) {
        *reinterpret_cast<uint4*>(&Xs[buf][lr][lc]) = rx0;
        *reinterpret_cast<uint4*>(&Xs[buf][lr][lc + 8]) = rx1;
        *reinterpret_cast<uint4*>(&Gs[buf][lr][lc]) = rg0;
        *reinterpret_cast<uint4*>(&Gs[buf][lr][lc + 8]) = rg1;
    };
    float acc[8][4];
#pragma unroll
    for (int i = 0; i < 8; ++i) acc[i][0] = acc[i][1] = acc[i][2] = acc[i][3] = 0.0f;
    const int nst = (int)((e1 - e0 + kWS - 1) / kWS);
    const int r = lane & 7, mat = lane >> 3;
    fetch(e0);
    stash(0);
    __syncthreads();
    for (int st = 0; st < nst; ++st) {
        const int cur = st & 1;
        if (st + 1 < nst) fetch(e0 + (long long)(st + 1) * kWS);
#pragma unroll
        for (int kk = 0; kk < kWS; kk += 16) {
            // A (rows = input channels of this warp): matrices (m0, k0) = (0,0), (8,0), (0,8), (8,8)
            uint32_t a0, a1, a2, a3;
            ldsm_x4_t(a0, a1, a2, a3, &Xs[cur][kk + (mat >> 1) * 8 + r][warp * 16 + (mat & 1) * 8]);
#pragma unroll
            for (int np = 0; np < 4; ++np) {
                if (np * 16 < ncols) {
                    // B for column tiles 2np and 2np+1: matrices (k0, n0) = (0,0), (8,0), (0,8), (8,8)
                    uint32_t b0, b1, b2, b3;
                    ldsm_x4_t(b0, b1, b2, b3, &Gs[cur][kk + (mat & 1) * 8 + r][np * 16 + (mat >> 1) * 8]);
                    mma16816(acc[2 * np], a0, a1, a2, a3, b0, b1);
                    if ((2 * np + 1) * 8 < ncols) mma16816(acc[2 * np + 1], a0, a1, a2, a3, b2, b3);
                }
            }
        }
        if (st + 1 < nst) stash(cur ^ 1);
        __syncthreads();
    }
    const int g = lane >> 2, t = lane & 3;
#pragma unroll
    for (int nt = 0; nt < 8; ++nt) {
        const int co = co0 + nt * 8 + 2 * t;
        if (co >= a.Cout) continue;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int ci = ci0 + warp * 16 + g + 8 * h;
            if (ci >= a.Cin) continue;
            float* d = a.dw + ((size_t)tap * a.Cin + ci) * a.Cout + co;
            atomicAdd(d, acc[nt][2 * h]);
            atomicAdd(d + 1, acc[nt][2 * h + 1]);
        }
    }
}

// dbias[c] += sum over voxels of dy[.][c]: a block sums `block_rows` voxels, a thread 8 channels
// (16 bytes) of every (256 / (C / 8))-th of them; blockIdx.y: blocks of 2048 channels
constexpr int kBiasCh = 2048;
__global__ void __launch_bounds__(256) k_bias_grad(const bf16* __restrict__ dy, float* __restrict__ db, long long total,
                                                   int C, int block_rows)
{
    __shared__ float part[256][8];
    const int c0 = blockIdx.y * kBiasCh, Cb = min(C - c0, kBiasCh);
    const int C8 = Cb / 8, rows = 256 / C8;
    const int j = threadIdx.x % C8, r = threadIdx.x / C8;
    float s[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    if (r < rows) {
        const long long e0 = (long long)blockIdx.x * block_rows;
        const int n = (int)(total - e0 < block_rows ? total - e0 : block_rows);
        const uint4* p = reinterpret_cast<const uint4*>(dy + (size_t)e0 * C + c0) + j;
#pragma unroll 4
        for (int e = r; e < n; e += rows) {
            float f[8];
            unpack8(__ldg(p + (size_t)e * (C / 8)), f);
#pragma unroll
            for (int c = 0; c < 8; ++c) s[c] += f[c];
        }
    }
#pragma unroll
    for (int c = 0; c < 8; ++c) part[threadIdx.x][c] = s[c];
    __syncthreads();
    for (int c = threadIdx.x; c < Cb; c += 256) {
        float t = 0.0f;
        for (int k = 0; k < rows; ++k) t += part[k * C8 + c / 8][c % 8];
        atomicAdd(db + c0 + c, t);
    }
}

// pooling / upsampling over one BF16 channel pair per thread
__global__ void k_pool2(const bf16* __restrict__ x, bf16* __restrict__ y, int B, int D, int H, int W, int C)
{
    const int d = D / 2, h = H / 2, w = W / 2, C2 = C / 2;
    const long long n = (long long)B * d * h * w * C2;
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int c = (int)(i % C2) * 2;
    long long r = i / C2;
    const int xo = (int)(r % w), yo = (int)((r / w) % h), zo = (int)((r / ((long long)w * h)) % d);
    const int b = (int)(r / ((long long)w * h * d));
    float s0 = 0.0f, s1 = 0.0f;
    for (int k = 0; k < 8; ++k) {
        const int xs = 2 * xo + (k & 1), ys = 2 * yo + ((k >> 1) & 1), zs = 2 * zo + (k >> 2);
        const __nv_bfloat162 v = *reinterpret_cast<const __nv_bfloat162*>(
            x + ((((size_t)b * D + zs) * H + ys) * W + xs) * C + c);
        s0 += __low2float(v);
        s1 += __high2float(v);
    }
    *reinterpret_cast<__nv_bfloat162*>(y + (size_t)r * C + c) = __floats2bfloat162_rn(s0 * 0.125f, s1 * 0.125f);
}

// fine-grid pass: every fine voxel reads its coarse parent (pool gradient / upsampling)
template <bool kPoolGrad>
__global__ void k_fine_from_coarse(const bf16* __restrict__ src, bf16* __restrict__ dst, int B, int D, int H, int W,
                                   int C)
{
    // D, H, W: coarse sizes
    const int Df = 2 * D, Hf = 2 * H, Wf = 2 * W, C2 = C / 2;
    const long long n = (long long)B * Df * Hf * Wf * C2;
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int c = (int)(i % C2) * 2;
    const long long r = i / C2;
    const int xf = (int)(r % Wf), yf = (int)((r / Wf) % Hf), zf = (int)((r / ((long long)Wf * Hf)) % Df);
    const int b = (int)(r / ((long long)Wf * Hf * Df));
    const size_t p = ((((size_t)b * D + zf / 2) * H + yf / 2) * W + xf / 2) * C + c;
    __nv_bfloat162 v = *reinterpret_cast<const __nv_bfloat162*>(src + p);
    if (kPoolGrad) v = __floats2bfloat162_rn(__low2float(v) * 0.125f, __high2float(v) * 0.125f);
    *reinterpret_cast<__nv_bfloat162*>(dst + (size_t)r * C + c) = v;
}

// coarse-grid pass: sum of the 8 children (upsampling gradient)
__global__ void k_up2_grad(const bf16* __restrict__ dy, bf16* __restrict__ dx, int B, int D, int H, int W, int C)
{
    const int C2 = C / 2;
    const long long n = (long long)B * D * H * W * C2;
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int c = (int)(i % C2) * 2;
    const long long r = i / C2;
    const int xo = (int)(r % W), yo = (int)((r / W) % H), zo = (int)((r / ((long long)W * H)) % D);
    const int b = (int)(r / ((long long)W * H * D));
    const int Hf = 2 * H, Wf = 2 * W, Df = 2 * D;
    float s0 = 0.0f, s1 = 0.0f;
    for (int k = 0; k < 8; ++k) {
        const int xs = 2 * xo + (k & 1), ys = 2 * yo + ((k >> 1) & 1), zs = 2 * zo + (k >> 2);
        const __nv_bfloat162 v = *reinterpret_cast<const __nv_bfloat162*>(
            dy + ((((size_t)b * Df + zs) * Hf + ys) * Wf + xs) * C + c);
        s0 += __low2float(v);
        s1 += __high2float(v);
    }
    *reinterpret_cast<__nv_bfloat162*>(dx + (size_t)r * C + c) = __floats2bfloat162_rn(s0, s1);
}

// The same passes with 16-byte accesses: a thread has one coarse voxel and 8 channels, reads or
// writes its eight children. HBM-bound; with 4-byte accesses and 64-bit divisions per value they
// ran at 8-40 % of the measured bandwidth (up2 of 64^3 x 64 channels 493 us).
enum CoarseOp { kPool, kPoolGrad, kUp, kUpGrad, kPoolGradRelu, kUpGradRelu };

// src: the fine grid for kPool, kUpGrad(Relu), else the coarse one. kPoolGradRelu: dst[child] =
// (g[child] + src[parent] / 8) where act[child] > 0, else 0 (both BF16 roundings of the separate
// passes), and dst may be g: neither is restrict, and a thread reads its eight values of g, by
// ordinary loads, before it writes any. kUpGradRelu: dst[parent] = sum of the children where
// act[parent] > 0, else 0
template <int kOp>
__global__ void __launch_bounds__(256) k_coarse8(const bf16* __restrict__ src, const bf16* g,
                                                 const bf16* __restrict__ act, bf16* dst, unsigned n, int D, int H,
                                                 int W, int C8)
{
    // D, H, W: coarse sizes; n: coarse voxels of the batch x C8
    const unsigned i = blockIdx.x * 256u + threadIdx.x;
    if (i >= n) return;
    const unsigned r = i / (unsigned)C8, c = i - r * (unsigned)C8;
    const unsigned l = r / (unsigned)W, x = r - l * (unsigned)W;
    const unsigned q = l / (unsigned)H, y = l - q * (unsigned)H;  // q = b D + z
    const size_t f0 = (((size_t)(2 * q) * (2 * H) + 2 * y) * (2 * W) + 2 * x) * C8 + c;
    auto child = [&](int k) {
        return f0 + (((size_t)(k >> 2) * (2 * H) + (size_t)((k >> 1) & 1)) * (2 * W) + (size_t)(k & 1)) * C8;
    };
    const uint4* s = reinterpret_cast<const uint4*>(src);
    uint4* d = reinterpret_cast<uint4*>(dst);
    if constexpr (kOp == kPool || kOp == kUpGrad || kOp == kUpGradRelu) {
        float t[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        uint4 v[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) v[k] = __ldg(s + child(k));
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            float f[8];
            unpack8(v[k], f);
#pragma unroll
            for (int e = 0; e < 8; ++e) t[e] += f[e];
        }
        if constexpr (kOp == kPool) {
#pragma unroll
            for (int e = 0; e < 8; ++e) t[e] *= 0.125f;
        }
        if constexpr (kOp == kUpGradRelu) {
            float a[8];
            unpack8(__ldg(reinterpret_cast<const uint4*>(act) + i), a);
#pragma unroll
            for (int e = 0; e < 8; ++e) t[e] = a[e] > 0.0f ? t[e] : 0.0f;
        }
        d[i] = pack8(t);
    } else {
        uint4 v = __ldg(s + i);
        float p[8];
        if constexpr (kOp == kPoolGrad || kOp == kPoolGradRelu) {
            unpack8(v, p);
#pragma unroll
            for (int e = 0; e < 8; ++e) p[e] *= 0.125f;
            v = pack8(p);
            unpack8(v, p);  // rounded, as the separate pass stores it
        }
        uint4 gv[8];
        if constexpr (kOp == kPoolGradRelu) {
#pragma unroll
            for (int k = 0; k < 8; ++k) gv[k] = reinterpret_cast<const uint4*>(g)[child(k)];
        }
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const size_t o = child(k);
            if constexpr (kOp == kPoolGradRelu) {
                float gf[8], af[8];
                unpack8(gv[k], gf);
                unpack8(__ldg(reinterpret_cast<const uint4*>(act) + o), af);
#pragma unroll
                for (int e = 0; e < 8; ++e) gf[e] = af[e] > 0.0f ? gf[e] + p[e] : 0.0f;
                d[o] = pack8(gf);
            } else {
                d[o] = v;
            }
        }
    }
}

bool aligned16(const void* a, const void* b = nullptr, const void* c = nullptr, const void* d = nullptr)
{
    return (((uintptr_t)a | (uintptr_t)b | (uintptr_t)c | (uintptr_t)d) & 15) == 0;
}

// one pass of k_coarse8 where its 16-byte accesses and 32-bit index apply; false: use the
// general kernels (D, H, W: coarse sizes)
template <int kOp>
bool coarse8(const void* src, const void* g, const void* act, void* dst, int B, int D, int H, int W, int C,
             cudaStream_t s)
{
    const long long n = (long long)B * D * H * W * (C / 8);
    if (C % 8 || n >= (1LL << 31) || !aligned16(src, g, act, dst)) return false;
    k_coarse8<kOp><<<(unsigned)((n + 255) / 256), 256, 0, s>>>((const bf16*)src, (const bf16*)g, (const bf16*)act,
                                                               (bf16*)dst, (unsigned)n, D, H, W, C / 8);
    return true;
}

// y = a + b, or (kRelu) y[i] = b[i] where a[i] > 0, else 0 (y may alias either): eight values a
// thread (16 bytes) where `vec`, the rest one by one
template <bool kRelu>
__global__ void __launch_bounds__(256) k_pair(const bf16* a, const bf16* b, bf16* y, long long n, int vec)
{
    const long long i = (long long)blockIdx.x * 256 + threadIdx.x;
    const long long n8 = vec ? n / 8 : 0;
    if (i < n8) {
        float p[8], q[8];
        unpack8(reinterpret_cast<const uint4*>(a)[i], p);
        unpack8(reinterpret_cast<const uint4*>(b)[i], q);
#pragma unroll
        for (int e = 0; e < 8; ++e) q[e] = kRelu ? (p[e] > 0.0f ? q[e] : 0.0f) : p[e] + q[e];
        reinterpret_cast<uint4*>(y)[i] = pack8(q);
    } else if (i < n8 + (n - 8 * n8)) {
        const long long e = 8 * n8 + (i - n8);
        const float p = __bfloat162float(a[e]), q = __bfloat162float(b[e]);
        y[e] = __float2bfloat16_rn(kRelu ? (p > 0.0f ? q : 0.0f) : p + q);
    }
}

// network coordinates (p, q, r) of lattice node (x, y, z) for a force along `axis`: the
// forced axis comes first, the other two keep their order
__device__ __forceinline__ void to_net(int axis, int x, int y, int z, int& p, int& q, int& r)
{
    if (axis == 0) {
        p = x; q = y; r = z;
    } else if (axis == 1) {
        p = y; q = x; r = z;
    } else {
        p = z; q = x; r = y;
    }
}
__device__ __forceinline__ void net_dims(int axis, int nx, int ny, int nz, int& P, int& Q, int& R)
{
    to_net(axis, nx, ny, nz, P, Q, R);
}
// lattice component of network channel c
__device__ __forceinline__ int lattice_comp(int axis, int c)
{
    if (axis == 0) return c;
    if (axis == 1) return c == 0 ? 1 : (c == 1 ? 0 : 2);
    return c == 0 ? 2 : (c == 1 ? 0 : 1);
}

// network voxel index (x fastest in network order: p fastest) of lattice node n
__device__ __forceinline__ int net_voxel(int axis, int n, int nx, int ny, int nz)
{
    const int x = n % nx, y = (n / nx) % ny, z = n / (nx * ny);
    int p, q, r, P, Q, R;
    to_net(axis, x, y, z, p, q, r);
    net_dims(axis, nx, ny, nz, P, Q, R);
    return (r * Q + q) * P + p;
}

__global__ void k_pack_input(const uint8_t* __restrict__ cls, bf16* __restrict__ x, int nx, int ny, int nz, int axis,
                             int vec)
{
    const int n = blockIdx.x * blockDim.x + threadIdx.x;
    const int N = nx * ny * nz;
    if (n >= N) return;
    const int v = net_voxel(axis, n, nx, ny, nz);
    const uint8_t c = cls[n];
    const uint32_t one = 0x3f80u;  // BF16 1
    const uint32_t w0 = ((c & 3) != 0 ? one : 0u) | ((c & 4) != 0 ? one << 16 : 0u);
    bf16* o = x + (size_t)v * 16;
    if (vec) {
        reinterpret_cast<uint4*>(o)[0] = make_uint4(w0, 0u, 0u, 0u);
        reinterpret_cast<uint4*>(o)[1] = make_uint4(0u, 0u, 0u, 0u);
    } else {
        unsigned short* h = reinterpret_cast<unsigned short*>(o);
        h[0] = (unsigned short)w0;
        h[1] = (unsigned short)(w0 >> 16);
        for (int k = 2; k < 16; ++k) h[k] = 0;
    }
}

// sum and count of y[.][3] over the forced cluster (FP64)
__global__ void __launch_bounds__(256) k_cluster_mean(const float* __restrict__ y, int ldy, const uint8_t* __restrict__ cls, int nx, int ny,
                               int nz, int axis, double* __restrict__ acc)
{
    const int N = nx * ny * nz;
    double s = 0.0;
    int c = 0;
    for (long long n = (long long)blockIdx.x * 256 + threadIdx.x; n < N; n += (long long)gridDim.x * 256) {
        if (cls[n] & 4) {
            s += y[(size_t)net_voxel(axis, (int)n, nx, ny, nz) * ldy + 3];
            ++c;
        }
    }
    // the block's sum, so that few atomic additions meet at the two totals
    __shared__ double part[8];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    const int cw = __reduce_add_sync(0xffffffffu, c);
    __shared__ int cnt[8];
    if ((threadIdx.x & 31) == 0) {
        part[threadIdx.x >> 5] = s;
        cnt[threadIdx.x >> 5] = cw;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        int k = 0;
        for (int w = 0; w < 8; ++w) {
            t += part[w];
            k += cnt[w];
        }
        if (k > 0) {
            atomicAdd(acc, t);
            atomicAdd(acc + 1, (double)k);
        }
    }
}

__global__ void k_unpack_output(const float* __restrict__ y, int ldy, const uint8_t* __restrict__ cls,
                                float* __restrict__ u, float* __restrict__ rho, int nx, int ny, int nz, int axis,
                                float scale_u, float scale_rho, const double* __restrict__ acc)
{
    const int n = blockIdx.x * blockDim.x + threadIdx.x;
    const int N = nx * ny * nz;
    if (n >= N || !(cls[n] & 4)) return;
    const int v = net_voxel(axis, n, nx, ny, nz);
    for (int c = 0; c < 3; ++c) u[(size_t)lattice_comp(axis, c) * N + n] += scale_u * y[(size_t)v * ldy + c];
    if (rho) {
        const float m = (float)(acc[0] / acc[1]);
        rho[n] += scale_rho * (y[(size_t)v * ldy + 3] - m);
    }
}

__global__ void k_pack_target(const float* __restrict__ u, const float* __restrict__ rho, float* __restrict__ t,
                              int nx, int ny, int nz, int axis, float scale_u, float scale_rho)
{
    const int n = blockIdx.x * blockDim.x + threadIdx.x;
    const int N = nx * ny * nz;
    if (n >= N) return;
    const int v = net_voxel(axis, n, nx, ny, nz);
    for (int c = 0; c < 3; ++c) t[(size_t)v * 4 + c] = scale_u * u[(size_t)lattice_comp(axis, c) * N + n];
    t[(size_t)v * 4 + 3] = rho[n] > 0.0f ? scale_rho * (rho[n] - 1.0f) : 0.0f;
}

// A thread takes whole voxels (16-byte accesses where `vec`: ldy a multiple of 8, four channels of
// targets, aligned); the block adds its FP64 sums before the one atomic addition
__global__ void __launch_bounds__(256) k_mse(const float* __restrict__ y, int ldy, const float* __restrict__ t, int nc,
                                             const bf16* __restrict__ x, bf16* __restrict__ dy,
                                             double* __restrict__ loss, long long total, double inv, int vec)
{
    double s = 0.0;
    const float scale = (float)(2.0 * inv);
    for (long long e = (long long)blockIdx.x * 256 + threadIdx.x; e < total; e += (long long)gridDim.x * 256) {
        const bool fluid = __bfloat162float(x[(size_t)e * 16]) > 0.5f;
        if (vec) {
            float g[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
            if (fluid) {
                const float4 a = *reinterpret_cast<const float4*>(y + (size_t)e * ldy);
                const float4 b = *reinterpret_cast<const float4*>(t + (size_t)e * 4);
                const float d[4] = {a.x - b.x, a.y - b.y, a.z - b.z, a.w - b.w};
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    s += (double)d[c] * d[c];
                    g[c] = scale * d[c];
                }
            }
            uint4* o = reinterpret_cast<uint4*>(dy + (size_t)e * ldy);
            o[0] = pack8(g);
            for (int c = 1; c < ldy / 8; ++c) o[c] = make_uint4(0u, 0u, 0u, 0u);
            continue;
        }
        for (int c = 0; c < ldy; ++c) {
            float gval = 0.0f;
            if (fluid && c < nc) {
                const float d = y[(size_t)e * ldy + c] - t[(size_t)e * nc + c];
                s += (double)d * d;
                gval = scale * d;
            }
            dy[(size_t)e * ldy + c] = __float2bfloat16_rn(gval);
        }
    }
    __shared__ double part[8];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        double b = 0.0;
        for (int w = 0; w < 8; ++w) b += part[w];
        if (b != 0.0) atomicAdd(loss, b * inv);
    }
}

__global__ void k_adam(float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m, float* __restrict__ v,
                       long long n, float lr, float b1, float b2, float eps, float c1, float c2, bf16* __restrict__ wf,
                       bf16* __restrict__ wb, int cin, int cout)
{
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.0f - b1) * gi;
    const float vi = b2 * v[i] + (1.0f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    const float pi = p[i] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    p[i] = pi;
    if (wf) {
        // master index (tap, ci, co) -> forward copy [tap][co][ci], transposed copy [tap][ci][co]
        const long long per = (long long)cin * cout;
        const int tap = (int)(i / per);
        const int ci = (int)((i % per) / cout), co = (int)(i % cout);
        const bf16 h = __float2bfloat16_rn(pi);
        wf[((size_t)tap * cout + co) * cin + ci] = h;
        wb[i] = h;
    }
}

// Tensor map of the weights [27][N][K] for boxes of NB output channels x 64 input channels
// (channels beyond K read as zero; 128-byte swizzle). False where the driver does not offer the
// encoder or refuses the address.
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
EncodeTiledFn tensor_map_encoder()
{
    static const EncodeTiledFn fn = [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) != cudaSuccess ||
            q != cudaDriverEntryPointSuccess) {
            (void)cudaGetLastError();
            p = nullptr;
        }
        return (EncodeTiledFn)p;
    }();
    return fn;
}

bool weight_map(const ConvArgs& a, int NB, CUtensorMap* map)
{
    const EncodeTiledFn encode = tensor_map_encoder();
    if (!encode) return false;
    const cuuint64_t dims[3] = {(cuuint64_t)a.K, (cuuint64_t)a.N, 27};
    const cuuint64_t strides[2] = {(cuuint64_t)a.K * 2, (cuuint64_t)a.K * a.N * 2};
    const cuuint32_t box[3] = {64, (cuuint32_t)NB, 1}, one[3] = {1, 1, 1};
    return encode(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<bf16*>(a.w), dims, strides, box, one,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Shape of the marching kernel for one layer, or false where it does not apply. The channel
// block NB and the strip length T are those with the least estimated time: waves of one unit
// per SM times the clocks of a unit, where a staged row costs the larger of its MMAs (products
// at 4096 per clock, operands at 128 bytes per clock), its copies (about 40 bytes per clock
// and SM from L2) and 250 clocks of hand-over.
bool march_plan(const ConvArgs& a, int B, int sms, MarchArgs* out, size_t* smem)
{
    const int K = a.K, N = a.N;
    if (!fills_groups(a.W) || !(K == 16 || K == 32 || K == 64 || K == 96 || K == 128) || (long long)B * a.V >= (1LL << 31)) return false;
    const int kch = (K + 63) / 64;
    const size_t abytes = (size_t)kch * kMChunk;
    MarchArgs best{};
    double best_cost = 0.0;
    size_t best_smem = 0;
    for (int nblk = 1; nblk * 16 <= N; ++nblk) {
        if (N % (16 * nblk)) continue;
        const int NB = N / nblk;
        if (3 * NB > 256) continue;
        const size_t bbytes = (size_t)3 * kch * 3 * NB * 128;
        const bool resident = nblk == 1 && 3 * bbytes + 3 * abytes <= (size_t)kMSmem - 1024;
        const size_t bsm = (resident ? 3 : 2) * bbytes;
        if (bsm + 2 * abytes > (size_t)kMSmem - 1024) continue;
        const int nA = (int)std::min<size_t>(kMStages, ((size_t)kMSmem - 1024 - bsm) / abytes);
        for (int T = 1; T <= a.H && T <= 16 && T * NB <= 512; T = T < 4 ? T + 1 : T + 2) {
            const int bufs = 2 * T * NB <= 512 ? 2 : 1;
            const int GX = (a.W + 7) / 8, NG = B * a.D * GX;
            const long long units = (long long)((NG + 15) / 16) * ((a.H + T - 1) / T) * nblk;
            if (units > (1LL << 30)) continue;
            double rows = 0.0;
            for (int r = 0; r < T + 2; ++r) {
                const int nn = (std::min(2, T + 1 - r) - std::max(0, 2 - r) + 1) * NB;
                const double mma = 3.0 * (K / 16) * std::max(nn / 2.0, 32.0 + nn / 4.0);
                rows += std::max(std::max(mma, kMRows * K * 2 / 40.0), 250.0);
            }
            const double unit = 3.0 * rows + (resident ? 0.0 : 3.0 * 9 * NB * K * 2 / 100.0) +
                                (bufs == 1 ? 8.0 * T * NB : 0.0) + 500.0;
            const double cost = (double)((units + sms - 1) / sms) * unit + 3000.0 + 8.0 * T * NB;
            if (best_cost == 0.0 || cost < best_cost) {
                best_cost = cost;
                best.c = a;
                best.GX = GX;
                best.NG = NG;
                best.T = T;
                best.nstrip = (a.H + T - 1) / T;
                best.NB = NB;
                best.nblk = nblk;
                best.units = (int)units;
                best.nA = nA;
                best.resident = resident ? 1 : 0;
                best.bufs = bufs;
                best.ncols = 32;
                while ((int)best.ncols < bufs * T * NB) best.ncols <<= 1;
                best_smem = bsm + nA * abytes + 1024;
            }
        }
    }
    if (best_cost == 0.0) return false;
    *out = best;
    *smem = best_smem;
    return true;
}

template <int kCI>
void (*wgrad_kernel(int co))(const WgradTcArgs)
{
    return co == 64 ? k_wgrad_tc<kCI, 64> : (co == 32 ? k_wgrad_tc<kCI, 32> : k_wgrad_tc<kCI, 16>);
}

int grid1(long long n, int block) { return (int)((n + block - 1) / block); }

}  // namespace

extern "C" {

static int conv3d(const void* x, const void* w, const float* bias, void* y, float* yf, void* y2, const void* other,
                  int mode, int up, int B, int D, int H, int W, int K, int N, int sign, int relu, void* stream)
{
    ConvArgs a{(const bf16*)x, (const bf16*)w, bias, (bf16*)y, yf, D, H, W, D * H * W, K, N, sign, relu != 0,
               (bf16*)y2, (const bf16*)other, mode, up != 0};
    const int bn = N < kTMaxN ? N : kTMaxN;
    int dev = 0, sms = 0;
    MP_CUDA(cudaGetDevice(&dev));
    MP_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    MarchArgs m;
    size_t msmem = 0;
    CUtensorMap wmap;
    if (march_plan(a, B, sms, &m, &msmem) && weight_map(a, m.NB, &wmap)) {
        void (*mkern)(const MarchArgs, const CUtensorMap) = K == 16   ? k_conv_march<16>
                                         : K == 32 ? k_conv_march<32>
                                         : K == 64 ? k_conv_march<64>
                                         : K == 96 ? k_conv_march<96>
                                                   : k_conv_march<128>;
        MP_CUDA(cudaFuncSetAttribute(mkern, cudaFuncAttributeMaxDynamicSharedMemorySize, kMSmem));
        mkern<<<std::min(m.units, sms), kMThreads, msmem, (cudaStream_t)stream>>>(m, wmap);
        MP_CUDA(cudaGetLastError());
        return MP_OK;
    }
    // the ring plus room to align it to a 1024-byte boundary
    const size_t smem = (size_t)kTStages * (kTABytes + (size_t)(bn / 8) * kTAtom) + kTAtom;
    // boxes narrower than three voxels, other channel counts, weights off a 16-byte boundary: tap by
    // tap, with the usual channel counts fixed at compile time
    void (*kern)(const ConvArgs) = K == 16   ? k_conv_tc<16>
                                   : K == 32 ? k_conv_tc<32>
                                   : K == 64 ? k_conv_tc<64>
                                   : K == 96 ? k_conv_tc<96>
                                   : K == 128 ? k_conv_tc<128>
                                               : k_conv_tc<0>;
    MP_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)(kTStages * (kTABytes + (kTMaxN / 8) * kTAtom) + kTAtom)));
    dim3 grid((a.V + kTM - 1) / kTM, (N + kTMaxN - 1) / kTMaxN, B);
    kern<<<grid, kTThreads, smem, (cudaStream_t)stream>>>(a);
    MP_CUDA(cudaGetLastError());
    return MP_OK;
}

static bool conv_args_ok(const void* x, const void* w, int B, int D, int H, int W, int K, int N, int sign)
{
    return x && w && B >= 1 && D >= 1 && H >= 1 && W >= 1 && K >= 16 && N >= 16 && K % 16 == 0 && N % 16 == 0 &&
           (sign == 1 || sign == -1) && (long long)D * H * W <= (1LL << 30);
}

int sg_conv3d(const void* x, const void* w, const float* bias, void* y, float* yf, int B, int D, int H, int W, int K,
              int N, int sign, int relu, void* stream)
{
    clear_error();
    if (!conv_args_ok(x, w, B, D, H, W, K, N, sign) || (!y && !yf)) {
        set_error("sg_conv3d: needs x, w, an output, B, D, H, W >= 1, K and N multiples of 16, sign +-1");
        return MP_EINVAL;
    }
    return conv3d(x, w, bias, y, yf, nullptr, nullptr, 0, 0, B, D, H, W, K, N, sign, relu, stream);
}

int sg_conv3d_ex(const void* x, const void* w, const float* bias, void* y, float* yf, void* y2, const void* other,
                 int mode, int up, int B, int D, int H, int W, int K, int N, int sign, int relu, void* stream)
{
    clear_error();
    if (!conv_args_ok(x, w, B, D, H, W, K, N, sign) || (!y && !yf && !y2) || mode < 0 || mode > 2 ||
        ((mode != 0) != (y2 != nullptr)) || ((mode != 0) != (other != nullptr)) || (up && (D % 2 || H % 2 || W % 2))) {
        set_error("sg_conv3d_ex: needs what sg_conv3d needs, y2 and other exactly with mode 1 or 2, and even D, H, W "
                  "with up");
        return MP_EINVAL;
    }
    return conv3d(x, w, bias, y, yf, y2, other, mode, up, B, D, H, W, K, N, sign, relu, stream);
}

int sg_check(void* stream)
{
    clear_error();
    int h = 0;
    MP_CUDA(cudaMemcpyFromSymbolAsync(&h, g_sg_tc_fail, sizeof(int), 0, cudaMemcpyDeviceToHost, (cudaStream_t)stream));
    MP_CUDA(cudaStreamSynchronize((cudaStream_t)stream));
    if (h) {
        const int zero = 0;
        MP_CUDA(cudaMemcpyToSymbolAsync(g_sg_tc_fail, &zero, sizeof(int), 0, cudaMemcpyHostToDevice, (cudaStream_t)stream));
        MP_CUDA(cudaStreamSynchronize((cudaStream_t)stream));
        set_error("sg_check: a bounded wait of the tensor-core convolution gave up (its output is not valid)");
        return MP_ETIMEOUT;
    }
    return MP_OK;
}

int sg_conv3d_wgrad(const void* x, const void* dy, float* dw, float* dbias, int B, int D, int H, int W, int Cin,
                    int Cout, void* stream)
{
    return sg_conv3d_wgrad_ex(x, dy, dw, dbias, 0, B, D, H, W, Cin, Cout, stream);
}

int sg_conv3d_wgrad_ex(const void* x, const void* dy, float* dw, float* dbias, int up, int B, int D, int H, int W,
                       int Cin, int Cout, void* stream)
{
    clear_error();
    if (!x || !dy || !dw || B < 1 || D < 1 || H < 1 || W < 1 || Cin < 16 || Cout < 16 || Cin % 16 || Cout % 16 ||
        (up && (D % 2 || H % 2 || W % 2))) {
        set_error("sg_conv3d_wgrad: needs x, dy, dw, positive sizes (even with up), Cin and Cout multiples of 16");
        return MP_EINVAL;
    }
    const int ci_tiles = (Cin + kWM - 1) / kWM, co_tiles = (Cout + kWN - 1) / kWN;
    WgradArgs a{(const bf16*)x, (const bf16*)dy, dw, D, H, W, D * H * W, Cin, Cout, (long long)B * D * H * W, 2048,
                ci_tiles, up != 0};
    cudaStream_t cs = (cudaStream_t)stream;
    const long long nchunk = (a.total + a.chunk - 1) / a.chunk;
    int dev = 0, sms = 0;
    MP_CUDA(cudaGetDevice(&dev));
    MP_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    WgradTcArgs m{a.x, a.dy, a.dw, D, H, W, Cin, Cout, a.up, {}};
    // A unit of the tensor-core kernel adds up its partial sums for a whole column of 128 voxels; on the
    // smallest boxes the general kernel, one block a tap and channel tile, is done earlier. Both, us without
    // bias (general / tensor cores): 64 voxels, 64 -> 64 channels 6.4 / 10.8, 32 -> 32 4.7 / 6.8; 128
    // voxels 6.8 / 10.7, 6.5 / 6.8; 256 voxels 10.6 / 10.7, 8.8 / 6.8; 384 voxels 12.8 / 10.8, 10.8 / 6.8
    const bool few = a.total <= (channel_block(Cin) == 64 ? 256 : 128);
    const bool tc = !few && wgrad_plan(B, D, H, W, Cin, Cout, sms, &m.p);
    if (nchunk * 27 > 2147483647LL || ci_tiles * co_tiles > 65535) {
        set_error("sg_conv3d_wgrad: too many voxels or channels");
        return MP_EINVAL;
    }
    if (tc) {
        const int ci = channel_block(Cin), co = channel_block(Cout);
        auto kern = ci == 64 ? wgrad_kernel<64>(co) : (ci == 32 ? wgrad_kernel<32>(co) : wgrad_kernel<16>(co));
        MP_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kMSmem - 1024));
        kern<<<std::min(m.p.units, sms), kGThreads, m.p.smem, cs>>>(m);
    } else {
        dim3 grid((unsigned)(nchunk * 27), (unsigned)(ci_tiles * co_tiles));
        k_wgrad<<<grid, kWThreads, 0, cs>>>(a);
    }
    MP_CUDA(cudaGetLastError());
    if (dbias) {
        // two blocks an SM, of 64 to 1024 voxels: in blocks of 1024 the four of a 64 x 64 x 1 box with 256
        // channels took 11 us longer
        const int rows = (int)std::min<long long>(1024, std::max<long long>(64, (a.total + 2 * sms - 1) / (2 * sms)));
        k_bias_grad<<<dim3(grid1(a.total, rows), (Cout + kBiasCh - 1) / kBiasCh), 256, 0, cs>>>((const bf16*)dy, dbias,
                                                                                              a.total, Cout, rows);
        MP_CUDA(cudaGetLastError());
    }
    return MP_OK;
}

int sg_pool2(const void* x, void* y, int B, int D, int H, int W, int C, void* stream)
{
    clear_error();
    if (!x || !y || B < 1 || D < 2 || H < 2 || W < 2 || (D | H | W) & 1 || C < 2 || C & 1) {
        set_error("sg_pool2: needs even D, H, W and an even channel count");
        return MP_EINVAL;
    }
    if (coarse8<kPool>(x, nullptr, nullptr, y, B, D / 2, H / 2, W / 2, C, (cudaStream_t)stream)) {
        MP_CUDA(cudaGetLastError());
        return MP_OK;
    }
    const long long n = (long long)B * (D / 2) * (H / 2) * (W / 2) * (C / 2);
    k_pool2<<<grid1(n, 256), 256, 0, (cudaStream_t)stream>>>((const bf16*)x, (bf16*)y, B, D, H, W, C);
    MP_CUDA(cudaGetLastError());
    return MP_OK;
}

int sg_pool2_grad(const void* dy, void* dx, int B, int D, int H, int W, int C, void* stream)
{
    clear_error();
    if (!dy || !dx || B < 1 || D < 2 || H < 2 || W < 2 || (D | H | W) & 1 || C < 2 || C & 1) {
        set_error("sg_pool2_grad: needs even D, H, W and an even channel count");
        return MP_EINVAL;
    }
    if (coarse8<kPoolGrad>(dy, nullptr, nullptr, dx, B, D / 2, H / 2, W / 2, C, (cudaStream_t)stream)) {
        MP_CUDA(cudaGetLastError());
        return MP_OK;
    }
    const long long n = (long long)B * D * H * W * (C / 2);
    k_fine_from_coarse<true><<<grid1(n, 256), 256, 0, (cudaStream_t)stream>>>((const bf16*)dy, (bf16*)dx, B, D / 2,
                                                                               H / 2, W / 2, C);
    MP_CUDA(cudaGetLastError());
    return MP_OK;
}

int sg_up2(const void* x, void* y, int B, int D, int H, int W, int C, void* stream)
{
    clear_error();
    if (!x || !y || B < 1 || D < 1 || H < 1 || W < 1 || C < 2 || C & 1) {
        set_error("sg_up2: needs positive sizes and an even channel count");
        return MP_EINVAL;
    }
    if (coarse8<kUp>(x, nullptr, nullptr, y, B, D, H, W, C, (cudaStream_t)stream)) {
        MP_CUDA(cudaGetLastError());
        return MP_OK;
    }
    const long long n = (long long)B * 8 * D * H * W * (C / 2);
    k_fine_from_coarse<false><<<grid1(n, 256), 256, 0, (cudaStream_t)stream>>>((const bf16*)x, (bf16*)y, B, D, H, W,
                                                                                C);
    MP_CUDA(cudaGetLastError());
    return MP_OK;
}

int sg_up2_grad(const void* dy, void* dx, int B, int D, int H, int W, int C, void* stream)
{
    clear_error();
    if (!dy || !dx || B < 1 || D < 1 || H < 1 || W < 1 || C < 2 || C & 1) {
        set_error("sg_up2_grad: needs positive sizes and an even channel count");
        return MP_EINVAL;
    }
    if (coarse8<kUpGrad>(dy, nullptr, nullptr, dx, B, D, H, W, C, (cudaStream_t)stream)) {
        MP_CUDA(cudaGetLastError());
        return MP_OK;
    }
    const long long n = (long long)B * D * H * W * (C / 2);
    k_up2_grad<<<grid1(n, 256), 256, 0, (cudaStream_t)stream>>>((const bf16*)dy, (bf16*)dx, B, D, H, W, C);
    MP_CUDA(cudaGetLastError());
    return MP_OK;
}

int sg_up2_grad_relu(const void* dy, const void* act, void* dx, int B, int D, int H, int W, int C, void* stream)
{
    clear_error();
    if (!dy || !act || !dx || B < 1 || D < 1 || H < 1 || W < 1 || C < 8 || C % 8) {
        set_error("sg_up2_grad_relu: needs positive sizes and a channel count that is a multiple of 8");
        return MP_EINVAL;
    }
    if (!coarse8<kUpGradRelu>(dy, nullptr, act, dx, B, D, H, W, C, (cudaStream_t)stream)) {
        set_error("sg_up2_grad_relu: buffers must be 16-byte aligned, with less than 2^34 values");
        return MP_EINVAL;
    }
    MP_CUDA(cudaGetLastError());
    return MP_OK;
}

int sg_pool2_grad_relu(const void* dy, const void* g, const void* act, void* dx, int B, int D, int H, int W, int C,
                       void* stream)
{
    clear_error();
    if (!dy || !g || !act || !dx || B < 1 || D < 2 || H < 2 || W < 2 || (D | H | W) & 1 || C < 8 || C % 8) {
        set_error("sg_pool2_grad_relu: needs even D, H, W and a channel count that is a multiple of 8");
        return MP_EINVAL;
    }
    if (!coarse8<kPoolGradRelu>(dy, g, act, dx, B, D / 2, H / 2, W / 2, C, (cudaStream_t)stream)) {
        set_error("sg_pool2_grad_relu: buffers must be 16-byte aligned, with less than 2^34 values");
        return MP_EINVAL;
    }
    MP_CUDA(cudaGetLastError());
    return MP_OK;
}

int sg_add(const void* a, const void* b, void* y, int64_t n, void* stream)
{
    clear_error();
    if (!a || !b || !y || n < 0) {
        set_error("sg_add: NULL pointer or negative count");
        return MP_EINVAL;
    }
    if (n == 0) return MP_OK;
    const int vec = aligned16(a, b, y);
    k_pair<false><<<grid1(vec ? n / 8 + n % 8 : n, 256), 256, 0, (cudaStream_t)stream>>>((const bf16*)a, (const bf16*)b,
                                                                                         (bf16*)y, n, vec);
    MP_CUDA(cudaGetLastError());
    return MP_OK;
}

int sg_relu_grad(const void* act, void* g, int64_t n, void* stream)
{
    clear_error();
    if (!act || !g || n < 0) {
        set_error("sg_relu_grad: NULL pointer or negative count");
        return MP_EINVAL;
    }
    if (n == 0) return MP_OK;
    const int vec = aligned16(act, g);
    k_pair<true><<<grid1(vec ? n / 8 + n % 8 : n, 256), 256, 0, (cudaStream_t)stream>>>(
        (const bf16*)act, (const bf16*)g, (bf16*)g, n, vec);
    MP_CUDA(cudaGetLastError());
    return MP_OK;
}

int sg_pack_input(const uint8_t* cls, void* x, int nx, int ny, int nz, int axis, void* stream)
{
    clear_error();
    if (!cls || !x || nx < 1 || ny < 1 || nz < 1 || axis < 0 || axis > 2) {
        set_error("sg_pack_input: bad arguments");
        return MP_EINVAL;
    }
    const int N = nx * ny * nz;
    k_pack_input<<<grid1(N, 256), 256, 0, (cudaStream_t)stream>>>(cls, (bf16*)x, nx, ny, nz, axis, aligned16(x));
    MP_CUDA(cudaGetLastError());
    return MP_OK;
}

int sg_unpack_output(const float* y, int ldy, const uint8_t* cls, float* u, float* rho, int nx, int ny, int nz,
                     int axis, float scale_u, float scale_rho, void* stream)
{
    clear_error();
    if (!y || !cls || !u || ldy < (rho ? 4 : 3) || nx < 1 || ny < 1 || nz < 1 || axis < 0 || axis > 2) {
        set_error("sg_unpack_output: bad arguments");
        return MP_EINVAL;
    }
    cudaStream_t s = (cudaStream_t)stream;
    const int N = nx * ny * nz;
    double* acc = nullptr;
    if (rho) {
        MP_CUDA(pool_malloc((void**)&acc, 2 * sizeof(double), s));
        cudaError_t e = cudaMemsetAsync(acc, 0, 2 * sizeof(double), s);
        if (e == cudaSuccess) {
            k_cluster_mean<<<std::min(grid1(N, 256), 152 * 8), 256, 0, s>>>(y, ldy, cls, nx, ny, nz, axis, acc);
            e = cudaGetLastError();
        }
        if (e != cudaSuccess) {
            cudaFreeAsync(acc, s);
            return cuda_fail(e, "sg_unpack_output");
        }
    }
    k_unpack_output<<<grid1(N, 256), 256, 0, s>>>(y, ldy, cls, u, rho, nx, ny, nz, axis, scale_u, scale_rho, acc);
    cudaError_t e = cudaGetLastError();
    if (acc) cudaFreeAsync(acc, s);
    if (e != cudaSuccess) return cuda_fail(e, "sg_unpack_output");
    return MP_OK;
}

int sg_pack_target(const float* u, const float* rho, float* t, int nx, int ny, int nz, int axis, float scale_u,
                   float scale_rho, void* stream)
{
    clear_error();
    if (!u || !rho || !t || nx < 1 || ny < 1 || nz < 1 || axis < 0 || axis > 2) {
        set_error("sg_pack_target: bad arguments");
        return MP_EINVAL;
    }
    const int N = nx * ny * nz;
    k_pack_target<<<grid1(N, 256), 256, 0, (cudaStream_t)stream>>>(u, rho, t, nx, ny, nz, axis, scale_u, scale_rho);
    MP_CUDA(cudaGetLastError());
    return MP_OK;
}

int sg_mse(const float* y, int ldy, const float* t, int nc, const void* x, void* dy, double* loss, int B, int V,
           double n_fluid, void* stream)
{
    clear_error();
    if (!y || !t || !x || !dy || !loss || nc < 1 || nc > ldy || B < 1 || V < 1 || !(n_fluid > 0.0)) {
        set_error("sg_mse: bad arguments");
        return MP_EINVAL;
    }
    const long long total = (long long)B * V;
    const int vec = ldy % 8 == 0 && nc == 4 && aligned16(y, t, dy);
    const int blocks = (int)std::min<long long>((total + 255) / 256, 152 * 16);
    k_mse<<<blocks, 256, 0, (cudaStream_t)stream>>>(y, ldy, t, nc, (const bf16*)x, (bf16*)dy, loss, total,
                                                    1.0 / (nc * n_fluid), vec);
    MP_CUDA(cudaGetLastError());
    return MP_OK;
}

int sg_adam(float* p, const float* g, float* m, float* v, int64_t n, float lr, float b1, float b2, float eps, int t,
            void* wf, void* wb, int cin, int cout, void* stream)
{
    clear_error();
    if (!p || !g || !m || !v || n < 0 || t < 1 || ((wf != nullptr) != (wb != nullptr)) ||
        (wf && (cin < 1 || cout < 1 || n != 27LL * cin * cout))) {
        set_error("sg_adam: bad arguments (weights need n = 27 cin cout and both copies)");
        return MP_EINVAL;
    }
    if (n == 0) return MP_OK;
    const float c1 = 1.0f - powf(b1, (float)t), c2 = 1.0f - powf(b2, (float)t);
    k_adam<<<grid1(n, 256), 256, 0, (cudaStream_t)stream>>>(p, g, m, v, n, lr, b1, b2, eps, c1, c2, (bf16*)wf,
                                                             (bf16*)wb, cin, cout);
    MP_CUDA(cudaGetLastError());
    return MP_OK;
}

}  // extern "C"
