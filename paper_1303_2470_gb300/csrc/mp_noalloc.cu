// mp_noalloc.cu -- one moment-propagation + sorption step on caller-owned dense arrays that
// allocates no memory at all, for callers that cannot allocate device memory: code that runs
// inside a host application which owns every device allocation (a fixed memory budget or
// its own pool, where a stray cudaMalloc would fail or break its accounting), or code that
// must not trigger the implicit device synchronisation of cudaMalloc / cudaFree.
//
// The only scratch the step needs -- the per-block partial sums of its FP64 reduction -- lives
// in a file-scope __device__ array of fixed size. Every GPU that runs this entry point keeps
// that array until the library is unloaded.
#include <mutex>

#include "internal.cuh"
#include "lattice.cuh"
#include "link_arith.cuh"

using namespace mp;

namespace {

constexpr int kNaThreads = 128;
constexpr int kNaNodes = 256;       // nodes per block
constexpr int kNaMaxBlocks = 8192;  // at most 2,097,152 nodes per call
constexpr long long kNaMaxNodes = (long long)kNaNodes * kNaMaxBlocks;

// one FP64 partial sum per block
static __device__ __align__(256) unsigned char g_noalloc_scratch[kNaMaxBlocks * sizeof(double)];

struct NaArgs {
    int nx, ny, nz, N;
    int g;  // direction of the velocity weight of the sum, -1 for the plain sum
    float hl, pa, pd;
    Div dx, dxy;  // division by nx and by nx*ny
};

// Same update as the library's step kernel, read from dense arrays: X(r) + sum of net link
// fluxes, then the sorption exchange on interfacial nodes (paper Sec. "Algorithm",
// Eqs. propagated_quantity, Pads, newP), and sum_r X'(r) u*_g(r) in FP64.
// Everything is recomputed from the mask and the flow, about 1270 instructions a fluid node, and in
// a porous medium most lanes of a warp of consecutive nodes are solid. So a block packs the fluid
// nodes of its 256 onto its 128 threads (in one or two rounds), with 64 registers and no branch around
// a link, so that the loads of several links are in flight; the sums are taken over the nodes in
// their own order all the same. A call on 64^3 spheres (porosity 0.4) takes 14.3 us (one thread a
// node, a branch a link: 20.8), on 127^3 51 us (93). What bounds it now: issuing takes 3.3 us of
// 64^3 and half the time of 127^3; the 64^3 launch is 0.84 of a wave with 40 % of the issue slots
// used, and waits on its chain (mask bytes, packing, two barriers, eighteen mask bytes, the
// gathers) and then for the sum's launch.
template <bool kFlow>
__global__ void __launch_bounds__(kNaThreads, 8)
    k_step_noalloc(const __grid_constant__ NaArgs a, const uint8_t* __restrict__ solid, const float* __restrict__ u,
                   const float* __restrict__ X, const float* __restrict__ Xa, float* __restrict__ Xn,
                   float* __restrict__ Xan, unsigned char* __restrict__ scratch)
{
    double* partials = reinterpret_cast<double*>(scratch);
    cudaTriggerProgrammaticLaunchCompletion();
    constexpr int kRounds = kNaNodes / kNaThreads;
    __shared__ float s_z[kNaNodes];
    __shared__ unsigned char s_list[kNaNodes];  // the block's fluid nodes, ascending
    __shared__ int s_count[kNaNodes / 32];
    const int base = blockIdx.x * kNaNodes;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    bool fl[kRounds];
    uint32_t bits[kRounds];
#pragma unroll
    for (int r = 0; r < kRounds; ++r) {
        const int l = r * kNaThreads + threadIdx.x, n = base + l;
        fl[r] = n < a.N && solid[n] == 0;
        bits[r] = __ballot_sync(0xffffffffu, fl[r]);
        if (lane == 0) s_count[r * (kNaThreads / 32) + warp] = __popc(bits[r]);
        s_z[l] = 0.0f;
        if (n < a.N && !fl[r]) {
            Xn[n] = 0.0f;
            Xan[n] = 0.0f;
        }
    }
    __syncthreads();
    int total = 0;
#pragma unroll
    for (int w = 0; w < kNaNodes / 32; ++w) total += s_count[w];
#pragma unroll
    for (int r = 0; r < kRounds; ++r) {
        int before = 0;
        for (int w = 0; w < r * (kNaThreads / 32) + warp; ++w) before += s_count[w];
        if (fl[r]) s_list[before + __popc(bits[r] & ((1u << lane) - 1u))] = (unsigned char)(r * kNaThreads + threadIdx.x);
    }
    __syncthreads();
    for (int j = threadIdx.x; j < total; j += kNaThreads) {
        const int l = s_list[j], n = base + l;
        const Nbr b = nbrs_of(a.nx, a.ny, a.nz, a.dx, a.dxy, n);
        float ux = 0.f, uy = 0.f, uz = 0.f;
        if (kFlow) {
            ux = u[n];
            uy = u[a.N + n];
            uz = u[2 * a.N + n];
        }
        const float ar = rn_mul(-1.5f, rn_add(rn_add(rn_mul(ux, ux), rn_mul(uy, uy)), rn_mul(uz, uz)));
        const float whl_face = rn_mul(weight<float>(1), a.hl), whl_edge = rn_mul(weight<float>(5), a.hl);
        const float xr = X[n];
        float delta = 0.0f, us = 0.0f;
        uint32_t mask = 0;
#pragma unroll
        for (int i = 1; i < kQ; ++i) mask |= (__ldg(solid + src_of(b, i)) == 0 ? 1u : 0u) << (i - 1);
#pragma unroll
        for (int i = 1; i < kQ; ++i) {
            const int s = src_of(b, i);
            const bool open = (mask >> (i - 1)) & 1u;
            float sx = 0.f, sy = 0.f, sz = 0.f;
            if (kFlow) {
                sx = (open ? __ldg(u + s) : 0.0f);
                sy = (open ? __ldg(u + a.N + s) : 0.0f);
                sz = (open ? __ldg(u + 2 * a.N + s) : 0.0f);
            }
            const float xs = (open ? __ldg(X + s) : 0.0f);
            const float as = rn_mul(-1.5f, rn_add(rn_add(rn_mul(sx, sx), rn_mul(sy, sy)), rn_mul(sz, sz)));
            const float whl = is_face(i) ? whl_face : whl_edge;
            const float pin = rn_fma(weight<float>(i), qlink(edot<float>(i, sx, sy, sz), as), whl);
            const float pout = rn_fma(weight<float>(i), qlink(edot<float>(opposite(i), ux, uy, uz), ar), whl);
            const float d = rn_add(delta, rn_sub(rn_mul(pin, xs), rn_mul(pout, xr)));
            delta = open ? d : delta;
            if (a.g >= 0) {
                const int c = ci(opposite(i), a.g);
                if (c != 0) us += open ? float(c) * pout : 0.0f;
            }
        }
        if (mask != (1u << (kQ - 1)) - 1u) {
            const float xa = Xa[n];
            const float js = rn_sub(rn_mul(a.pa, xr), rn_mul(a.pd, xa));
            delta = rn_sub(delta, js);
            Xan[n] = rn_add(xa, js);
        } else {
            Xan[n] = 0.0f;
        }
        const float xn = rn_add(xr, delta);
        Xn[n] = xn;
        s_z[l] = a.g >= 0 ? xn * us : xn;
    }
    __syncthreads();
    // FP32 within 32 consecutive nodes, FP64 across them and blocks, in a fixed order
    __shared__ double s_red[kNaNodes / 32];
#pragma unroll
    for (int r = 0; r < kRounds; ++r) {
        float zp = s_z[r * kNaThreads + threadIdx.x];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) zp += __shfl_xor_sync(0xffffffffu, zp, o);
        if (lane == 0) s_red[r * (kNaThreads / 32) + warp] = (double)zp;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < kNaNodes / 32; ++w) t += s_red[w];
        partials[blockIdx.x] = t;
    }
}

// The sum of the block partials, in a fixed order. A launch of its own (programmatic dependent
// launch: resident by the time the step ends) in place of a completion counter, which had to be
// cleared by a launch before the step and made its last block work alone.
__global__ void __launch_bounds__(256) k_sum_noalloc(const double* __restrict__ partials, int blocks,
                                                     double* __restrict__ z_out)
{
    __shared__ double s_w[8];
    cudaGridDependencySynchronize();
    double v = 0.0;
    for (int b = threadIdx.x; b < blocks; b += 256) v += __ldcg(partials + b);
    v = warp_sum(v);
    if ((threadIdx.x & 31) == 0) s_w[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < 8; ++w) t += s_w[w];
        *z_out = t;
    }
}

// Device address of the scratch array. In host code the array's name is only a host-side
// stand-in, so the address is looked up with cudaGetSymbolAddress (with the device current)
// and remembered per device together with the unique id of the context it belongs to. A
// cudaDeviceReset ends that context and the next call runs in a new one, whose module copy
// of the array lives elsewhere: a changed context id triggers a fresh lookup.
std::mutex g_scratch_mu;
struct ScratchSlot {
    unsigned char* ptr = nullptr;
    unsigned long long ctx_id = 0;
};
ScratchSlot g_scratch[128];

int scratch_address(unsigned char** out)
{
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return cuda_fail(e, "cudaGetDevice");
    if (dev < 0 || dev >= 128) {
        set_error("mp_step_noalloc: device ordinal out of range");
        return MP_EINVAL;
    }
    std::lock_guard<std::mutex> lock(g_scratch_mu);
    ScratchSlot& slot = g_scratch[dev];
    const unsigned long long id = slot.ptr ? current_ctx_id() : 0;
    if (!slot.ptr || id == 0 || id != slot.ctx_id) {
        void* p = nullptr;
        e = cudaGetSymbolAddress(&p, g_noalloc_scratch);  // also makes the device's context current
        if (e != cudaSuccess) return cuda_fail(e, "cudaGetSymbolAddress(scratch)");
        slot.ptr = static_cast<unsigned char*>(p);
        slot.ctx_id = current_ctx_id();
    }
    *out = slot.ptr;
    return MP_OK;
}

// [a, a + na) and [b, b + nb) share a byte (null pointers share nothing)
bool overlap(const void* a, size_t na, const void* b, size_t nb)
{
    if (!a || !b || na == 0 || nb == 0) return false;
    const uintptr_t x = reinterpret_cast<uintptr_t>(a), y = reinterpret_cast<uintptr_t>(b);
    return x < y + nb && y < x + na;
}

}  // namespace

extern "C" int mp_step_noalloc(int nx, int ny, int nz, const uint8_t* solid, const float* u, double D_b,
                               double k_a, double k_d, int direction, const float* X, const float* X_ads,
                               float* X_out, float* X_ads_out, double* Z_out, void* stream)
{
    clear_error();
    if (nx < 3 || ny < 3 || nz < 3) {
        set_error("mp_step_noalloc: every lattice dimension must be >= 3");
        return MP_EINVAL;
    }
    const long long N = (long long)nx * ny * nz;
    if (N > kNaMaxNodes) {
        set_error("mp_step_noalloc: " + std::to_string(N) + " nodes exceed the limit of " +
                  std::to_string(kNaMaxNodes) + " set by its fixed reduction scratch");
        return MP_EINVAL;
    }
    if (!solid || !X || !X_ads || !X_out || !X_ads_out || !Z_out) {
        set_error("mp_step_noalloc: solid, X, X_ads, X_out, X_ads_out and Z_out are required");
        return MP_EINVAL;
    }
    {
        // the step reads neighbours of every node while other threads write their results,
        // so no output byte may lie in any input (or in the other output)
        const size_t fb = (size_t)N * sizeof(float);
        const void* in[5] = {X, X_ads, solid, u, Z_out};
        const size_t in_b[5] = {fb, fb, (size_t)N, u ? 3 * fb : 0, sizeof(double)};
        const void* outs[2] = {X_out, X_ads_out};
        bool bad = overlap(X_out, fb, X_ads_out, fb);
        for (int o = 0; o < 2; ++o)
            for (int j = 0; j < 5; ++j) bad = bad || overlap(outs[o], fb, in[j], in_b[j]);
        if (bad) {
            set_error("mp_step_noalloc: the output arrays must not overlap the inputs, Z_out or each other");
            return MP_EINVAL;
        }
    }
    if (!(D_b > 0.0 && D_b <= 0.25) || !(k_a >= 0.0 && k_a <= 1.0) || !(k_d >= 0.0 && k_d <= 1.0) ||
        direction < -1 || direction > 2) {
        set_error("mp_step_noalloc: need 0 < D_b <= 0.25, k_a and k_d in [0, 1], direction in -1..2");
        return MP_EINVAL;
    }
    unsigned char* scratch = nullptr;
    int rc = scratch_address(&scratch);
    if (rc != MP_OK) return rc;
    cudaStream_t s = (cudaStream_t)stream;
    NaArgs a;
    a.nx = nx;
    a.ny = ny;
    a.nz = nz;
    a.N = (int)N;
    a.g = direction;
    a.hl = (float)(6.0 * D_b);  // lambda/2 = 12 D_b / 2
    a.pa = (float)k_a;
    a.pd = (float)k_d;
    const int blocks = (int)((N + kNaNodes - 1) / kNaNodes);
    a.dx = make_div((unsigned)nx);
    a.dxy = make_div((unsigned)(nx * ny));
    auto kern = u ? k_step_noalloc<true> : k_step_noalloc<false>;
    kern<<<blocks, kNaThreads, 0, s>>>(a, solid, u, X, X_ads, X_out, X_ads_out, scratch);
    MP_CUDA(cudaGetLastError());
    MP_CUDA(launch_pdl(k_sum_noalloc, dim3(1), dim3(256), s, (const double*)scratch, blocks, Z_out));
    return MP_OK;
}
