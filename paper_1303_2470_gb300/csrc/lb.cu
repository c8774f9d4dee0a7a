// lb.cu -- steady BGK lattice-Boltzmann flow (paper Eq. lb_evolution) for the velocity
// field that biases the moment propagation. One fused pull step per launch:
//   stream   f_i(r) <- f_i^post(r - c_i), or f_ibar^post(r) when r - c_i is solid
//            (halfway bounce-back, ibar the opposite link);
//   moments  rho = sum f_i, u = (sum f_i c_i + F/2) / rho;
//   collide  f_i^post = f_i - (f_i - f_i^eq(rho,u))/tau
//                       + (1 - 1/(2 tau)) w_i [3 (c_i - u) + 9 (c_i.u) c_i].F   (Guo force).
// Populations are FP32 deviations g_i = f_i - w_i, which keeps ~9 significant digits of the
// O(u) part that sets the velocity, stored for fluid nodes only, in the order of the sorted
// fluid list: g[i*N_F + k] for fluid node k (structure of arrays). One thread per fluid node;
// the compact index of a neighbour s is prefix[s >> 5] + popc(fluid bits of s's word below
// s), from two bit-sized arrays that stay cache-resident, so a warp's reads and writes cover
// whole sectors of fluid data only. The steady criterion max|u(t) - u(t-1)| is evaluated
// without rounding.
// The body force acts on the largest connected fluid cluster only (sealed pockets stay at
// rest, their steady Stokes velocity). At every failed residual check the state is replaced
// by the mean of the last two iterates: the fixed point is unchanged, an error mode of
// eigenvalue lambda is scaled by (1 + lambda)/2, and the undamped period-2 modes that
// bounce-back sustains at nodes with few open links disappear (without it the residual of a
// porous medium stalls near |F|).
#include <cfloat>
#include <cmath>
#include <cstring>
#include <string>

#include "internal.cuh"
#include "lattice.cuh"

using namespace mp;

namespace {

// Blocks of 128 threads, 10 per SM (48 registers a thread): the step keeps its 19 gathers and
// their places in registers. Measured per step at 128^3 / 192^3 / 384^3: 26.5 / 80.8 / 645 us; 256 x 5
// 26.7 / 81.7 / 656, 256 x 4 28.6 / 87.9 / 734, 512 x 2 30.4 / 92.0 / 781. Launches that a SM's share of
// 1024 threads takes in one wave (kLbSmall nodes) run blocks of 64 with 64 registers: nothing
// waits for a block slot, small blocks spread evenly (64^3: 4.2 us, 5.0 with 128 x 10).
constexpr int kLbThreads = 128, kLbMinBlocks = 10;
constexpr int kLbSmallThreads = 64, kLbSmallMinBlocks = 16;
constexpr long long kLbSmall = 152LL * 1024;

struct LbArgs {
    int nx, ny, nz, N, NF;
    Div dx, dxy;  // division by nx and by nx*ny
    const uint32_t* fluid;
    const int32_t* fbase;    // fluid nodes before each 32-node word
    const int32_t* flist;    // lattice node of fluid index k
    const uint32_t* omask;   // fluid index k: bit i-1: r - c_i is fluid; kXlo, kXhi, kForced
    const uint4* rows;       // fluid index k: eight 16-bit offsets of the row centres from k
    const uint2* fw;         // {fluid bits, fluid nodes before the word} per 32-node word
    const uint32_t* forced;  // the force acts on these nodes (the largest fluid cluster)
    float Fx, Fy, Fz;
    float inv_tau;
    float guo;  // 1 - 1/(2 tau)
};

// |a - b| of two FP32 numbers without rounding, as a key that orders like the value: the FP32
// difference s and its rounding error e (a - b = s + e exactly; Knuth's two-sum), the bits of |s|
// above those of e towards |s| made to order as unsigned. In FP64 the same comparison took some
// 35 operations of a pipe that does two per clock and SM (50 us of a 128^3 check).
__device__ __forceinline__ unsigned long long diff_key(float a, float b)
{
    const float s = __fsub_rn(a, b), t = __fsub_rn(s, a);
    float e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, t)), __fsub_rn(-b, t));
    if (s < 0.0f) e = -e;
    const uint32_t w = __float_as_uint(e);
    return ((unsigned long long)__float_as_uint(fabsf(s)) << 32) | (w ^ ((w >> 31) ? 0xffffffffu : 0x80000000u));
}
double key_value(unsigned long long key)
{
    const uint32_t sb = (uint32_t)(key >> 32);
    uint32_t eb = (uint32_t)key;
    eb = (eb >> 31) ? eb ^ 0x80000000u : ~eb;
    float s, e;
    memcpy(&s, &sb, 4);
    memcpy(&e, &eb, 4);
    return key == 0 ? 0.0 : (std::isfinite(s) ? (double)s + (double)e : (double)INFINITY);
}

// flags beside the 18 link bits: x - 1 and x + 1 lie in the node's row without wrapping, the
// force acts on the node
constexpr uint32_t kXlo = 1u << 18, kXhi = 1u << 19, kForced = 1u << 20;
constexpr int kFarRow = -32768;  // a row centre out of the 16-bit offsets' reach

__device__ __forceinline__ bool lb_bit(const uint32_t* __restrict__ w, int n)
{
    return (__ldg(w + (n >> 5)) >> (n & 31)) & 1u;
}

// mode 0: plain step; 1: also store u into u_prev; 2: store u into u_out (and rho into
// rho_out when given), fold max|u - u_prev| into *res_key (diff_key), then store u into
// u_prev. u_prev is compact [3][N_F]; u_out and rho_out are dense (their solid entries are
// zeroed once by the host).
// Everything static (the sources' places) is worked out before griddepcontrol.wait, while the
// previous step drains. kRows: the row centres come as 16-bit offsets from a table of 16 bytes
// a node instead of eight lookups (about 100 of 870 instructions; the step issues 70 % of the
// time); rows beyond their reach, where z wraps around, are looked up. kWide: populations
// beyond 2^32 elements (a source's plane is then found at its load).
template <bool kRows, bool kWide, int kB, int kMinBlocks>
__global__ void __launch_bounds__(kB, kMinBlocks)
    k_lb_step(const __grid_constant__ LbArgs a, const float* g_in, float* __restrict__ gn, int mode, float* u_prev_in,
              float* __restrict__ u_out, float* __restrict__ rho_out,
              unsigned long long* __restrict__ res_key)
{
    cudaTriggerProgrammaticLaunchCompletion();
    const int k = blockIdx.x * kB + threadIdx.x;
    const size_t NF = (size_t)a.NF;
    unsigned long long res = 0;
    const bool active = k < a.NF;
    const uint32_t nf = (uint32_t)a.NF;
    uint32_t at[kQ];  // element of g that link i is read from (kWide: without its plane)
    uint32_t mask = 0;
    if (active) {
        mask = __ldg(a.omask + k);
        // fluid-list index of each source row's centre; sources in a row are consecutive
        int C[8];
        if constexpr (kRows) {
            const uint4 r = __ldg(a.rows + k);
            const uint32_t w[4] = {r.x, r.y, r.z, r.w};
            bool far = false;
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const int o = (int)(short)(w[j >> 1] >> (16 * (j & 1)));
                C[j] = k + o;
                far |= o == kFarRow;
            }
            if (far) {
                const Nbr b = nbrs_of(a.nx, a.ny, a.nz, a.dx, a.dxy, __ldg(a.flist + k));
#pragma unroll
                for (int j = 0; j < 8; ++j) C[j] = fluid_index(a.fw, src_of(b, row_centre(j)));
            }
        } else {
            const Nbr b = nbrs_of(a.nx, a.ny, a.nz, a.dx, a.dxy, __ldg(a.flist + k));
#pragma unroll
            for (int j = 0; j < 8; ++j) C[j] = fluid_index(a.fw, src_of(b, row_centre(j)));
        }
        at[0] = (uint32_t)k;
#pragma unroll
        for (int i = 1; i < kQ; ++i) {
            const int row = row_of(i);
            const int base = row < 0 ? k : C[row < 0 ? 0 : row];
            int s = base;
            if (cx(i) > 0) s = base - 1;
            if (cx(i) < 0) s = base + (row < 0 ? 1 : (int)((mask >> (row_centre(row < 0 ? 0 : row) - 1)) & 1u));
            const bool open = (mask >> (i - 1)) & 1u;  // else halfway bounce-back
            at[i] = (open ? (uint32_t)s : (uint32_t)k) + (kWide ? 0u : (open ? (uint32_t)i : (uint32_t)opposite(i)) * nf);
        }
        if ((mask & (kXlo | kXhi)) != (kXlo | kXhi)) {
            // the sources beyond the wrap of x (rare) are looked up one by one
            const Nbr b = nbrs_of(a.nx, a.ny, a.nz, a.dx, a.dxy, __ldg(a.flist + k));
#pragma unroll
            for (int i = 1; i < kQ; ++i)
                if (cx(i) != 0 && !(mask & (cx(i) > 0 ? kXlo : kXhi)) && ((mask >> (i - 1)) & 1u))
                    at[i] = (uint32_t)fluid_index(a.fw, src_of(b, i)) + (kWide ? 0u : (uint32_t)i * nf);
        }
    }
    cudaGridDependencySynchronize();  // the previous step's populations and residual are visible
    const float* g = after_wait(g_in);
    float* u_prev = after_wait(u_prev_in);
    if (active) {
        float f[kQ];
#pragma unroll
        for (int i = 0; i < kQ; ++i) {
            const size_t plane = kWide ? (size_t)(i == 0 || ((mask >> (i > 0 ? i - 1 : 0)) & 1u) ? i : opposite(i)) * NF : 0;
            f[i] = g[plane + at[i]];
        }
        // the reference of a check, read before the 19 stores: behind them the three loads waited
        // for the stores to drain (135 us instead of 33 for a checked step of a 128^3 box)
        float px = 0.f, py = 0.f, pz = 0.f;
        if (mode == 2) {
            px = u_prev[k];
            py = u_prev[NF + k];
            pz = u_prev[2 * NF + k];
        }
        float drho = 0.f, mx = 0.f, my = 0.f, mz = 0.f;
#pragma unroll
        for (int i = 0; i < kQ; ++i) {
            drho += f[i];
            mx += float(cx(i)) * f[i];
            my += float(cy(i)) * f[i];
            mz += float(cz(i)) * f[i];
        }
        const bool on = (mask & kForced) != 0;
        const float Fx = on ? a.Fx : 0.0f, Fy = on ? a.Fy : 0.0f, Fz = on ? a.Fz : 0.0f;
        const float rho = 1.0f + drho;
        const float inv_rho = 1.0f / rho;
        const float ux = (mx + 0.5f * Fx) * inv_rho;
        const float uy = (my + 0.5f * Fy) * inv_rho;
        const float uz = (mz + 0.5f * Fz) * inv_rho;
        const float uu = ux * ux + uy * uy + uz * uz;
        const float uF = ux * Fx + uy * Fy + uz * Fz;
        const float m15uu = -1.5f * uu;
        const float m3uF = -3.0f * uF;
#pragma unroll
        for (int i = 0; i < kQ; ++i) {
            const float w = weight<float>(i);
            // c_i.u and c_i.F: signed sums of one or two components (zero for the rest link)
            float cu = 0.f, cF = 0.f;
            if (cx(i)) {
                cu += float(cx(i)) * ux;
                cF += float(cx(i)) * Fx;
            }
            if (cy(i)) {
                cu += float(cy(i)) * uy;
                cF += float(cy(i)) * Fy;
            }
            if (cz(i)) {
                cu += float(cz(i)) * uz;
                cF += float(cz(i)) * Fz;
            }
            // f^eq - w = w [(rho - 1) + rho (cu (3 + 4.5 cu) - 1.5 uu)]
            const float geq = w * fmaf(rho, fmaf(cu, fmaf(4.5f, cu, 3.0f), m15uu), drho);
            // Guo: (1 - 1/(2 tau)) w [3 (c_i - u).F + 9 (c_i.u)(c_i.F)] = ... w [3 cF (1 + 3 cu) - 3 u.F]
            const float src = a.guo * w * fmaf(3.0f * cF, fmaf(3.0f, cu, 1.0f), m3uF);
            gn[(size_t)i * NF + k] = fmaf(-a.inv_tau, f[i] - geq, f[i]) + src;
        }
        if (mode == 1) {
            u_prev[k] = ux;
            u_prev[NF + k] = uy;
            u_prev[2 * NF + k] = uz;
        } else if (mode == 2) {
            const int n = __ldg(a.flist + k);
            u_out[n] = ux;
            u_out[(size_t)a.N + n] = uy;
            u_out[2 * (size_t)a.N + n] = uz;
            if (rho_out) rho_out[n] = rho;
            res = max(diff_key(ux, px), max(diff_key(uy, py), diff_key(uz, pz)));
            // a non-finite velocity counts as an infinite residual
            if (!(fabsf(ux) <= FLT_MAX && fabsf(uy) <= FLT_MAX && fabsf(uz) <= FLT_MAX)) res = 0x7f800000ull << 32;
            // this node's u(t) is the reference of the next check when it is due next step
            u_prev[k] = ux;
            u_prev[NF + k] = uy;
            u_prev[2 * NF + k] = uz;
        }
    }
    if (mode == 2) {
        // one atomic maximum per block, and only where it still raises the total (every warp's
        // met at one address: 110 us of a 128^3 step)
        __shared__ unsigned long long s_res[kB / 32];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) res = max(res, __shfl_xor_sync(0xffffffffu, res, o));
        if ((threadIdx.x & 31) == 0) s_res[threadIdx.x >> 5] = res;
        __syncthreads();
        if (threadIdx.x == 0) {
            for (int w = 1; w < kB / 32; ++w) res = max(res, s_res[w]);
            if (res > *(volatile unsigned long long*)res_key) atomicMax(res_key, res);
        }
    }
}

// g0 <- (g0 + g1) / 2 over all populations: the mean of the last two iterates (four a thread;
// both arrays start on 256-byte boundaries)
__global__ void __launch_bounds__(256) k_lb_mean(float* __restrict__ g0, const float* __restrict__ g1, size_t count)
{
    const size_t i = blockIdx.x * (size_t)256 + threadIdx.x, n4 = count / 4;
    if (i < n4) {
        float4 a = reinterpret_cast<const float4*>(g0)[i];
        const float4 b = reinterpret_cast<const float4*>(g1)[i];
        a.x = 0.5f * (a.x + b.x);
        a.y = 0.5f * (a.y + b.y);
        a.z = 0.5f * (a.z + b.z);
        a.w = 0.5f * (a.w + b.w);
        reinterpret_cast<float4*>(g0)[i] = a;
    } else if (i < n4 + count % 4) {
        const size_t k = 4 * n4 + (i - n4);
        g0[k] = 0.5f * (g0[k] + g1[k]);
    }
}

// f = f^eq(rho0, u0) as deviations (u0 = 0 and rho0 = 1 when NULL; both dense); u_prev = u0
__global__ void k_lb_init(const LbArgs a, const float* __restrict__ u0, const float* __restrict__ rho0,
                          float* __restrict__ g, float* __restrict__ u_prev)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= a.NF) return;
    const size_t NF = (size_t)a.NF;
    const int n = __ldg(a.flist + k);
    float ux = 0.f, uy = 0.f, uz = 0.f, rho = 1.f;
    if (u0) {
        ux = u0[n];
        uy = u0[(size_t)a.N + n];
        uz = u0[2 * (size_t)a.N + n];
    }
    if (rho0) rho = rho0[n];
    const float uu = ux * ux + uy * uy + uz * uz;
#pragma unroll
    for (int i = 0; i < kQ; ++i) {
        const float cu = float(cx(i)) * ux + float(cy(i)) * uy + float(cz(i)) * uz;
        // f^eq - w = w [(rho - 1) + rho (3 cu + 4.5 cu^2 - 1.5 uu)]
        g[(size_t)i * NF + k] = weight<float>(i) * ((rho - 1.0f) + rho * (3.0f * cu + 4.5f * cu * cu - 1.5f * uu));
    }
    u_prev[k] = ux;
    u_prev[NF + k] = uy;
    u_prev[2 * NF + k] = uz;
}

}  // namespace

// Per lb_steady call: the {fluid bits, prefix} words that locate link sources in the fluid list,
// then (k_lb_prep) the open-link mask and flags of every fluid node and, when `rows` is given,
// its row offsets.
__global__ void k_lb_words(const LbArgs a, int W, uint2* __restrict__ fw)
{
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t < W) fw[t] = make_uint2(a.fluid[t], (uint32_t)a.fbase[t]);
}
__global__ void k_lb_prep(const LbArgs a, uint32_t* __restrict__ omask, uint4* __restrict__ rows)
{
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= a.NF) return;
    const int n = a.flist[t];
    const Nbr b = nbrs_of(a.nx, a.ny, a.nz, a.dx, a.dxy, n);
    uint32_t m = 0;
#pragma unroll
    for (int i = 1; i < kQ; ++i) {
        const int s = src_of(b, i);
        if ((a.fluid[s >> 5] >> (s & 31)) & 1u) m |= 1u << (i - 1);
    }
    if (b.oxm == -1) m |= kXlo;
    if (b.oxp == 1) m |= kXhi;
    if (lb_bit(a.forced, n)) m |= kForced;
    omask[t] = m;
    if (rows) {
        uint32_t w[4] = {0u, 0u, 0u, 0u};
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const int o = fluid_index(a.fw, src_of(b, row_centre(j))) - t;
            const int v = o > kFarRow && o < -kFarRow ? o : kFarRow;
            w[j >> 1] |= (uint32_t)(v & 0xffff) << (16 * (j & 1));
        }
        rows[t] = make_uint4(w[0], w[1], w[2], w[3]);
    }
}

extern "C" int lb_steady(const mp_geometry* geom, const double force[3], double tau, double tol, int64_t max_steps,
                         int64_t check_every, const float* u_init, const float* rho_init, float* u_out,
                         float* rho_out, int64_t* steps_out, double* residual_out, void* stream_ptr)
{
    clear_error();
    if (!force || !u_out || !(tau > 0.5) || max_steps < 1 || check_every < 1 || !(tol >= 0.0)) {
        set_error("lb_steady: need force, u_out, tau > 1/2, tol >= 0, max_steps >= 1, check_every >= 1");
        return MP_EINVAL;
    }
    cudaStream_t s = (cudaStream_t)stream_ptr;
    Geometry G;
    int rc = build_geometry(geom, s, true, true, &G);
    if (rc != MP_OK) return rc;
    // the body force acts on the largest connected fluid cluster: in a sealed pocket a
    // uniform force is balanced by pressure and the steady velocity is zero
    rc = build_cluster(&G, s, true, false);
    if (rc != MP_OK) {
        free_geometry(&G, s, true);
        cudaStreamSynchronize(s);
        return rc;
    }
    const size_t N = (size_t)G.N;
    const size_t NF = (size_t)(G.n_fluid > 0 ? G.n_fluid : 1);
    float *g0 = nullptr, *g1 = nullptr, *uprev = nullptr;
    uint32_t* omask = nullptr;
    uint2* fw = nullptr;
    uint4* rows = nullptr;
    // the row table where 16-bit offsets reach the neighbouring planes (at the fluid nodes of a
    // plane on average)
    const bool wide = kQ * (unsigned long long)NF >= (1ull << 32);
    bool use_rows = !wide && (double)G.n_fluid / G.nz * 1.2 + G.nx < 32000.0;
    unsigned long long* res_d = nullptr;
    cudaError_t e = pool_malloc((void**)&g0, sizeof(float) * kQ * NF, s);
    if (e == cudaSuccess) e = pool_malloc((void**)&omask, sizeof(uint32_t) * NF, s);
    if (e == cudaSuccess) e = pool_malloc((void**)&fw, sizeof(uint2) * (size_t)(G.W > 0 ? G.W : 1), s);
    if (e == cudaSuccess) e = pool_malloc((void**)&g1, sizeof(float) * kQ * NF, s);
    if (e == cudaSuccess) e = pool_malloc((void**)&uprev, sizeof(float) * 3 * NF, s);
    if (e == cudaSuccess) e = pool_malloc((void**)&res_d, sizeof(unsigned long long), s);
    // last, and only if there is room for it: a tenth more memory, which the step can do without
    if (e == cudaSuccess && use_rows && pool_malloc((void**)&rows, sizeof(uint4) * NF, s) != cudaSuccess) {
        (void)cudaGetLastError();
        rows = nullptr;
        use_rows = false;
    }
    // solid entries of the dense outputs stay zero; fluid entries are written at every check
    if (e == cudaSuccess) e = cudaMemsetAsync(u_out, 0, sizeof(float) * 3 * N, s);
    if (e == cudaSuccess && rho_out) e = cudaMemsetAsync(rho_out, 0, sizeof(float) * N, s);
    auto cleanup = [&]() {
        if (g0) cudaFreeAsync(g0, s);
        if (g1) cudaFreeAsync(g1, s);
        if (uprev) cudaFreeAsync(uprev, s);
        if (omask) cudaFreeAsync(omask, s);
        if (fw) cudaFreeAsync(fw, s);
        if (rows) cudaFreeAsync(rows, s);
        if (res_d) cudaFreeAsync(res_d, s);
        free_geometry(&G, s, true);
        cudaStreamSynchronize(s);
    };
    if (e != cudaSuccess) {
        rc = cuda_fail(e, "lb_steady allocation");
        cleanup();
        return rc;
    }
    LbArgs a;
    a.nx = G.nx;
    a.ny = G.ny;
    a.nz = G.nz;
    a.N = G.N;
    a.NF = (int)G.n_fluid;
    a.dx = make_div((unsigned)G.nx);
    a.dxy = make_div((unsigned)(G.nx * G.ny));
    a.fluid = G.fluid;
    a.fbase = G.fbase;
    a.flist = G.flist;
    a.omask = omask;
    a.rows = rows;
    a.fw = fw;
    a.forced = G.cluster;
    a.Fx = (float)force[0];
    a.Fy = (float)force[1];
    a.Fz = (float)force[2];
    a.inv_tau = (float)(1.0 / tau);
    a.guo = (float)(1.0 - 0.5 / tau);
    // one thread per fluid node (at least one block, so that a medium without fluid still
    // runs its checks: its residual is 0)
    const bool small = (long long)NF <= kLbSmall;
    const int threads = small ? kLbSmallThreads : kLbThreads;
    const int blocks = (int)((NF + threads - 1) / threads);
    auto kern = wide ? k_lb_step<false, true, kLbThreads, kLbMinBlocks>
                : small ? (use_rows ? k_lb_step<true, false, kLbSmallThreads, kLbSmallMinBlocks>
                                    : k_lb_step<false, false, kLbSmallThreads, kLbSmallMinBlocks>)
                        : (use_rows ? k_lb_step<true, false, kLbThreads, kLbMinBlocks>
                                    : k_lb_step<false, false, kLbThreads, kLbMinBlocks>);
    k_lb_words<<<(unsigned)((G.W + 255) / 256), 256, 0, s>>>(a, G.W, fw);
    k_lb_prep<<<(unsigned)((NF + 255) / 256), 256, 0, s>>>(a, omask, rows);
    k_lb_init<<<blocks, threads, 0, s>>>(a, u_init, rho_init, g0, uprev);
    e = cudaGetLastError();
    int64_t t = 0;
    double res = INFINITY;
    bool converged = false;
    while (e == cudaSuccess && t < max_steps) {
        const int64_t t1 = t + 1;
        int mode = 0;
        if (t1 % check_every == 0 || t1 == max_steps)
            mode = 2;
        else if ((t1 + 1) % check_every == 0 || t1 + 1 == max_steps)
            mode = 1;
        if (mode == 2) e = cudaMemsetAsync(res_d, 0, sizeof(unsigned long long), s);
        if (e == cudaSuccess)
            e = launch_pdl(kern, dim3(blocks), dim3(threads), s, a, (const float*)g0, g1, mode, uprev, u_out,
                           rho_out, res_d);
        float* tmp = g0;
        g0 = g1;
        g1 = tmp;
        t = t1;
        if (mode == 2 && e == cudaSuccess) {
            unsigned long long bits = 0;
            e = cudaMemcpyAsync(&bits, res_d, sizeof(bits), cudaMemcpyDeviceToHost, s);
            if (e == cudaSuccess) e = cudaStreamSynchronize(s);
            res = key_value(bits);
            if (res < tol) {
                converged = true;
                break;
            }
            if (std::isinf(res)) break;  // the flow is no longer finite: give up
            // the mean of the last two iterates (g0 = t, g1 = t-1): same fixed point, and the
            // undamped period-2 modes that bounce-back sustains at confined nodes vanish
            if (t < max_steps) {
                const size_t count = (size_t)kQ * NF;
                k_lb_mean<<<(unsigned)((count / 4 + count % 4 + 255) / 256), 256, 0, s>>>(g0, g1, count);
                e = cudaGetLastError();
            }
        }
    }
    if (e != cudaSuccess) {
        rc = cuda_fail(e, "lb_steady step");
        cleanup();
        return rc;
    }
    cleanup();
    if (steps_out) *steps_out = t;
    if (residual_out) *residual_out = res;
    if (!converged) {
        set_error(std::isinf(res) ? "lb_steady: the velocity became non-finite by step " + std::to_string(t) +
                                        " (unstable: tau, force or initial state)"
                                  : "lb_steady: residual " + std::to_string(res) + " above tol after " +
                                        std::to_string(t) + " steps");
        return MP_ENOTCONVERGED;
    }
    return MP_OK;
}
