// mp_flux64.cu -- the flux-form step of mp.cu for FP64 contexts with the link probabilities
// tabulated. Same update (Eq. propagated_quantity as X + sum of exactly antisymmetric link
// fluxes, Eqs. Pads and newP), same roundings of every probability and flux.
//
// What bounds it: FP64 arithmetic (2 fused multiply-adds per clock and SM on sm_103a, against
// 128 in FP32) and, on the slit-sized lattices that FP64 runs are for, the latency of one
// dependent launch per step. So, unlike in FP32,
//  * both probabilities of every link are read from a per-context table (16 bytes a link)
//    instead of being recomputed from the flow: 8 FP64 operations per link and moment pair
//    instead of about 20, and u*_g is tabulated too;
//  * up to 19456 nodes four lanes share a node (links l, l + 4, ...) in blocks of 16 nodes, so
//    that even a lattice of a few hundred nodes spreads over many SMs; beyond, a thread has a
//    node of one moment to itself and two share one of two or three moments (sharing leaves
//    lanes idle in the node's own update, but four fields of 18 neighbours fill the registers);
//  * everything static is loaded before griddepcontrol.wait, i.e. while the previous step
//    drains; a step's critical path is one gather of the neighbours, the arithmetic and the
//    store;
//  * the series of a step is appended by one extra block of the next launch (or by a closing
//    launch) instead of by the last block of its own.
// Measured per step (graph replay; recomputing step of mp.cu -> this one): slit of 3 x 3 x 100
// fluid nodes 26.9 -> 3.5 us (three species 75 -> 4.3; 26 such contexts side by side
// 104 -> 29.7); random spheres 32^3 (13 k fluid nodes) 30.6 -> 15.3, 64^3 74 -> 37.6
// (four lanes a node: 52.3), 128^3 520 -> 273 us, where 164 FP64 operations a node at the
// card's rate would take 238 us.
#include <algorithm>
#include <cstring>
#include <string>

#include "flux_run.cuh"
#include "internal.cuh"
#include "lattice.cuh"
#include "link_arith.cuh"
#include "mp_ctx.cuh"

namespace mp {

struct F64Args {
    int NF, N, NI, S, M, K;
    int SC;      // species per chunk of the field layout (1 for one species)
    int nblk;    // blocks of nodes
    const int32_t* flist;
    const int32_t* aidx;  // compact interface index, -1 off the interface
    const int32_t* src;   // source node of each link (at64), -1 where it is solid
    const double2* tab;   // one species: {p_in, p_out}; several: {q_in, q_out} (at64)
    const double* ust;    // [S M][NF] u*_g of every species and propagated direction
    double* part;         // [2][nblk][K] partial sums of the series, by step parity
    double* Z;
    double* D;
    long long* tdev;
    long long cap;
    double whf[MP_MAX_SPECIES], whe[MP_MAX_SPECIES], pa[MP_MAX_SPECIES], pd[MP_MAX_SPECIES];
};

struct Flux64 {
    F64Args a;
    int lanes = 4;  // lanes per node; blocks of 64 threads with four, else of 128
    int32_t* aidx = nullptr;
    int32_t* src = nullptr;
    double2* tab = nullptr;
    double* ust = nullptr;
    double* part = nullptr;
};

namespace {

constexpr int kSmallNodes = 152 * 16 * 8;  // eight blocks of 16 nodes per SM

// entry of link l (0..17) of work item k in the link tables: lanes of a warp read 16-byte
// entries of consecutive addresses, whether they share nodes (node-major) or not (32 nodes
// link by link)
__host__ __device__ __forceinline__ size_t at64(bool shared, int k, int l)
{
    return shared ? (size_t)k * (kQ - 1) + l : ((size_t)(k >> 5) * (kQ - 1) + l) * 32 + (k & 31);
}

// bit i - 1: link i is a face link (weight 1/18), else an edge link (1/36)
constexpr uint32_t face_links()
{
    uint32_t m = 0;
    for (int i = 1; i < kQ; ++i)
        if (is_face(i)) m |= 1u << (i - 1);
    return m;
}
constexpr uint32_t kFaceLinks = face_links();

// series of the step whose partials have parity `parity`: warp w adds series w, w + warps, ...
// over the blocks (FP64, fixed order) and appends Z and D at t + 1
template <int kB>
__device__ __forceinline__ void append64(const F64Args& a, int parity)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const long long t1 = *((volatile long long*)a.tdev) + 1;
    const double* part = a.part + (size_t)parity * a.nblk * a.K;
    for (int j = warp; j < a.K; j += kB / 32) {
        double v = 0.0;
        for (int b = lane; b < a.nblk; b += 32) v += __ldcg(part + (size_t)b * a.K + j);
        v = warp_sum(v);
        if (lane == 0) {
            a.Z[(size_t)j * a.cap + t1] = v;
            a.D[(size_t)j * a.cap + t1] = a.D[(size_t)j * a.cap + t1 - 1] + v;
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) *a.tdev = t1;
}

template <int FP>
__device__ __forceinline__ void ld_rec64(const double* p, double (&v)[FP])
{
#pragma unroll
    for (int f = 0; f < FP; f += 2) {
        const double2 d = *reinterpret_cast<const double2*>(p + f);
        v[f] = d.x;
        v[f + 1] = d.y;
    }
}
template <int FP>
__device__ __forceinline__ void st_rec64(double* p, const double (&v)[FP])
{
#pragma unroll
    for (int f = 0; f < FP; f += 2) *reinterpret_cast<double2*>(p + f) = make_double2(v[f], v[f + 1]);
}

// block (x, y): nodes x kB/kLanes .. of species y; block (nblk, 0) appends the previous step
template <int FP, bool kSingle, int kLanes, int kB>
__global__ void __launch_bounds__(kB)
    k_step64(const __grid_constant__ F64Args a, const double* P, double* Pn, const double* A_in, double* An, int parity,
             int pending)
{
    cudaTriggerProgrammaticLaunchCompletion();
    const int sp = (int)blockIdx.y;
    if ((int)blockIdx.x == a.nblk) {
        cudaGridDependencySynchronize();
        if (pending && sp == 0) append64<kB>(a, parity ^ 1);
        return;
    }
    constexpr int kLinksPerLane = (kQ - 1 + kLanes - 1) / kLanes;
    constexpr bool kShared = kLanes > 1;
    __shared__ double s_red[kB / 32][3];
    const int sub = threadIdx.x & (kLanes - 1);
    const int k = (int)blockIdx.x * (kB / kLanes) + (int)threadIdx.x / kLanes;
    const bool active = k < a.NF;
    // static data of the node and of this lane's links, loaded while the previous step drains
    int n = 0, ai = -1;
    int s[kLinksPerLane];
    double2 tb[kLinksPerLane];
    double us[3] = {0.0, 0.0, 0.0};
#pragma unroll
    for (int j = 0; j < kLinksPerLane; ++j) s[j] = -1;
    if (active) {
        n = __ldg(a.flist + k);
        ai = __ldg(a.aidx + k);
#pragma unroll
        for (int j = 0; j < kLinksPerLane; ++j) {
            const int l = sub + kLanes * j;
            if (l < kQ - 1) {
                s[j] = __ldg(a.src + at64(kShared, k, l));
                tb[j] = __ldg(a.tab + at64(kShared, k, l));
            }
        }
        if (sub == 0)
#pragma unroll
            for (int m = 0; m < 3; ++m)
                if (m < a.M) us[m] = __ldg(a.ust + (size_t)(sp * a.M + m) * a.NF + k);
    }
    // element (row, species) of the chunk-major fields
    const size_t stride = kSingle ? FP : (size_t)a.SC * FP;
    const size_t off = kSingle ? 0 : (size_t)(sp % a.SC) * FP;
    const size_t base = kSingle ? 0 : (size_t)(sp / a.SC) * a.N * stride + off;
    if constexpr (!kSingle) {
        const double whf = a.whf[sp], whe = a.whe[sp];
#pragma unroll
        for (int j = 0; j < kLinksPerLane; ++j) {
            const int l = sub + kLanes * j;
            if (l < kQ - 1 && s[j] >= 0) {
                const bool face = ((kFaceLinks >> l) & 1u) != 0;
                const double w = face ? weight<double>(1) : weight<double>(5), whl = face ? whf : whe;
                tb[j] = make_double2(rn_fma(w, tb[j].x, whl), rn_fma(w, tb[j].y, whl));
            }
        }
    }
    cudaGridDependencySynchronize();  // the previous step's fields and series are visible
    const double* Ps = after_wait(P) + base;
    const double* A = after_wait(A_in);
    double xr[FP], delta[FP];
#pragma unroll
    for (int f = 0; f < FP; ++f) xr[f] = delta[f] = 0.0;
    if (active) {
        double xs[kLinksPerLane][FP];
#pragma unroll
        for (int j = 0; j < kLinksPerLane; ++j)
            if (s[j] >= 0) ld_rec64<FP>(Ps + (size_t)s[j] * stride, xs[j]);
        ld_rec64<FP>(Ps + (size_t)n * stride, xr);
#pragma unroll
        for (int j = 0; j < kLinksPerLane; ++j)
            if (s[j] >= 0)
#pragma unroll
                for (int f = 0; f < FP; ++f)
                    delta[f] = rn_add(delta[f], rn_sub(rn_mul(tb[j].x, xs[j][f]), rn_mul(tb[j].y, xr[f])));
    }
    // the node's partial sums, one per lane
#pragma unroll
    for (int o = 1; o < kLanes; o <<= 1)
#pragma unroll
        for (int f = 0; f < FP; ++f) delta[f] += __shfl_xor_sync(0xffffffffu, delta[f], o);
    double zv[3] = {0.0, 0.0, 0.0};
    if (active && sub == 0) {
        if (ai >= 0) {
            const double pa = a.pa[sp], pd = a.pd[sp];
            const size_t ia = (kSingle ? 0 : (size_t)(sp / a.SC) * a.NI * stride + off) + (size_t)ai * stride;
            double xa[FP], xan[FP];
            ld_rec64<FP>(A + ia, xa);
#pragma unroll
            for (int f = 0; f < FP; ++f) {
                const double js = rn_sub(rn_mul(pa, xr[f]), rn_mul(pd, xa[f]));
                delta[f] = rn_sub(delta[f], js);
                xan[f] = rn_add(xa[f], js);
            }
            st_rec64<FP>(An + ia, xan);
        }
        double xn[FP];
#pragma unroll
        for (int f = 0; f < FP; ++f) xn[f] = rn_add(xr[f], delta[f]);
        st_rec64<FP>(Pn + base + (size_t)n * stride, xn);
#pragma unroll
        for (int m = 0; m < 3; ++m)
            if (m < a.M && 1 + m < FP) zv[m] = xn[(1 + m) < FP ? 1 + m : 0] * us[m];
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int m = 0; m < 3; ++m) {
        if (m < a.M) {
            double w = zv[m];
#pragma unroll
            for (int o = kLanes; o < 32; o <<= 1) w += __shfl_xor_sync(0xffffffffu, w, o);
            if (lane == 0) s_red[warp][m] = w;
        }
    }
    __syncthreads();
    if (threadIdx.x < a.M) {
        double t = 0.0;
#pragma unroll
        for (int w = 0; w < kB / 32; ++w) t += s_red[w][threadIdx.x];
        a.part[((size_t)parity * a.nblk + blockIdx.x) * a.K + sp * a.M + threadIdx.x] = t;
    }
}

// appends the series of the last step of a run
__global__ void __launch_bounds__(256) k_finish64(const __grid_constant__ F64Args a, int parity)
{
    pdl_enter();
    append64<256>(a, parity);
}

// Tables of one context: sources, {in, out} link values, interface indices, u*_g. The values
// are formed exactly as in the step of mp.cu.
// kOne: one species, whose links need not be kept.
template <bool kOne>
__global__ void k_tables64(const F64Args a, const uint32_t* __restrict__ fmask, const uint32_t* __restrict__ iface,
                           const int32_t* __restrict__ ibase, const Flow4<double>* __restrict__ u4, int nx, int ny,
                           int nz, Div dx, Div dxy, int d0, int d1, int d2, int32_t* __restrict__ aidx,
                           int32_t* __restrict__ src, double2* __restrict__ tab, double* __restrict__ ust, bool shared)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= a.NF) return;
    const int n = a.flist[k];
    const uint32_t mask = fmask[k];
    const Nbr b = nbrs_of(nx, ny, nz, dx, dxy, n);
    const Flow4<double> ur = u4[n];
    const int dir[3] = {d0, d1, d2};
    aidx[k] = mask != (1u << 18) - 1u ? ibase[n >> 5] + __popc(iface[n >> 5] & ((1u << (n & 31)) - 1u)) : -1;
    // the links and the first species once, then u*_g of the others from the links (64^3 with 16
    // species 202 us; with the links formed again for each species 428; one species 39)
    [[maybe_unused]] double qo[kQ];
    double us[3] = {0.0, 0.0, 0.0};
#pragma unroll
    for (int i = 1; i < kQ; ++i) {
        const size_t at = at64(shared, k, i - 1);
        if constexpr (!kOne) qo[i] = 0.0;
        if (!((mask >> (i - 1)) & 1u)) {
            src[at] = -1;
            tab[at] = make_double2(0.0, 0.0);
            continue;
        }
        const int s = src_of(b, i);
        const Flow4<double> uf = u4[s];
        const double qin = qlink(edot<double>(i, uf.x, uf.y, uf.z), uf.w);
        const double qout = qlink(edot<double>(opposite(i), ur.x, ur.y, ur.z), ur.w);
        if constexpr (!kOne) qo[i] = qout;
        const double whl = is_face(i) ? a.whf[0] : a.whe[0];
        const double pout = rn_fma(weight<double>(i), qout, whl);
        src[at] = s;
        tab[at] = kOne ? make_double2(rn_fma(weight<double>(i), qin, whl), pout) : make_double2(qin, qout);
#pragma unroll
        for (int m = 0; m < 3; ++m)
            if (m < a.M) us[m] += (double)ci(opposite(i), dir[m]) * pout;
    }
    for (int m = 0; m < a.M; ++m) ust[(size_t)m * a.NF + k] = us[m];
    for (int sp = 1; !kOne && sp < a.S; ++sp) {
        us[0] = us[1] = us[2] = 0.0;
        const double whf = a.whf[sp], whe = a.whe[sp];
#pragma unroll
        for (int i = 1; i < kQ; ++i) {
            if (!((mask >> (i - 1)) & 1u)) continue;
            const double pout = rn_fma(weight<double>(i), qo[i], is_face(i) ? whf : whe);
#pragma unroll
            for (int m = 0; m < 3; ++m)
                if (m < a.M) us[m] += (double)ci(opposite(i), dir[m]) * pout;
        }
        for (int m = 0; m < a.M; ++m) ust[(size_t)(sp * a.M + m) * a.NF + k] = us[m];
    }
}

template <int FP, bool kSingle, int kLanes, int kB>
cudaError_t launch64_t(mp_ctx* c, int pending, bool programmatic)
{
    const F64Args& a = c->flux64->a;
    const int s = c->cur;
    return launch_dependent(programmatic, k_step64<FP, kSingle, kLanes, kB>, dim3(a.nblk + 1, a.S), dim3(kB), c->stream, a,
                            (const double*)c->P[s], (double*)c->P[1 - s], (const double*)c->A[s],
                            (double*)c->A[1 - s], s, pending);
}

cudaError_t launch64(mp_ctx* c, int pending, bool prog)
{
    const bool small = c->flux64->lanes == 4;
    if (c->FP == 2) {
        if (c->S == 1) return small ? launch64_t<2, true, 4, 64>(c, pending, prog) : launch64_t<2, true, 1, 128>(c, pending, prog);
        return small ? launch64_t<2, false, 4, 64>(c, pending, prog) : launch64_t<2, false, 1, 128>(c, pending, prog);
    }
    if (c->S == 1) return small ? launch64_t<4, true, 4, 64>(c, pending, prog) : launch64_t<4, true, 2, 128>(c, pending, prog);
    return small ? launch64_t<4, false, 4, 64>(c, pending, prog) : launch64_t<4, false, 2, 128>(c, pending, prog);
}

}  // namespace

void flux64_free(mp_ctx* c)
{
    if (!c->flux64) return;
    cudaFree(c->flux64->aidx);
    cudaFree(c->flux64->src);
    cudaFree(c->flux64->tab);
    cudaFree(c->flux64->ust);
    cudaFree(c->flux64->part);
    delete c->flux64;
    c->flux64 = nullptr;
}

// Builds the tables of an FP64 flux context whose fields are initialised. They take 364 bytes
// per fluid node plus 8 per series; where that does not fit (tables_fit) or cannot be allocated, the
// context keeps the step of mp.cu, which recomputes the link terms (c->flux64 stays NULL).
int flux64_setup(mp_ctx* c)
{
    const size_t NF = (size_t)c->geo.n_fluid, K = (size_t)(c->S * c->M);
    const size_t rows = (NF + 31) / 32 * 32;  // whole groups of 32 in the link tables
    const size_t bytes = rows * (18 * (sizeof(double2) + sizeof(int32_t)) + sizeof(int32_t) + sizeof(double) * K);
    if (!tables_fit(bytes)) return MP_OK;
    Flux64* f = new (std::nothrow) Flux64();
    if (!f) return MP_OK;
    c->flux64 = f;
    f->lanes = NF <= (size_t)kSmallNodes ? 4 : (c->FP == 2 ? 1 : 2);
    F64Args& a = f->a;
    memset(&a, 0, sizeof(a));
    a.NF = (int)NF;
    a.N = c->geo.N;
    a.NI = (int)c->geo.n_iface;
    a.S = c->S;
    a.M = c->M;
    a.K = (int)K;
    a.SC = c->SC;
    const size_t per_block = (f->lanes == 4 ? 64 : 128) / f->lanes;
    a.nblk = (int)((NF + per_block - 1) / per_block);
    cudaError_t e = cudaMalloc(&f->aidx, sizeof(int32_t) * NF);
    if (e == cudaSuccess) e = cudaMalloc(&f->src, sizeof(int32_t) * 18 * rows);
    if (e == cudaSuccess) e = cudaMalloc(&f->tab, sizeof(double2) * 18 * rows);
    if (e == cudaSuccess) e = cudaMalloc(&f->ust, sizeof(double) * K * NF);
    if (e == cudaSuccess) e = cudaMalloc(&f->part, sizeof(double) * 2 * (size_t)a.nblk * K);
    if (e != cudaSuccess) {
        (void)cudaGetLastError();
        flux64_free(c);
        return MP_OK;
    }
    a.flist = c->geo.flist;
    a.aidx = f->aidx;
    a.src = f->src;
    a.tab = f->tab;
    a.ust = f->ust;
    a.part = f->part;
    a.Z = c->Z;
    a.D = c->D;
    a.tdev = c->tdev;
    a.cap = c->cap;
    for (int s = 0; s < c->S; ++s) {
        const double hl = 6.0 * c->Db[s];  // lambda/2 = 12 D_b / 2
        a.whf[s] = weight<double>(1) * hl;
        a.whe[s] = weight<double>(5) * hl;
        a.pa[s] = c->ka[s];
        a.pd[s] = c->kd[s];
    }
    auto tables = c->S == 1 ? k_tables64<true> : k_tables64<false>;
    tables<<<(unsigned)((NF + 127) / 128), 128, 0, c->stream>>>(
        a, c->fmask, c->geo.iface, c->geo.ibase, (const Flow4<double>*)c->u4, c->geo.nx, c->geo.ny, c->geo.nz,
        make_div((unsigned)c->geo.nx), make_div((unsigned)(c->geo.nx * c->geo.ny)), c->dir[0], c->dir[1], c->dir[2],
        f->aidx, f->src, f->tab, f->ust, f->lanes > 1);
    MP_CUDA(cudaGetLastError());
    c->tables_new = true;
    return MP_OK;
}

int flux64_step(mp_ctx* c, long long n)
{
    return run_flux(
        c, n, [&](int pending, bool programmatic) { return launch64(c, pending, programmatic); },
        [&](int parity) { return launch_pdl(k_finish64, dim3(1), dim3(256), c->stream, c->flux64->a, parity); });
}

}  // namespace mp
