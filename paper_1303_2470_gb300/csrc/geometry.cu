// geometry.cu -- node classification of a medium (solid S, fluid F, interfacial I subset of
// F: fluid nodes with at least one solid D3Q19 neighbour; paper Sec. "Algorithm", the three
// node classes of the Boltzmann weights) packed into per-32-node bit words, plus the
// exclusive prefix and the sorted list of interfacial nodes used to address the compact
// adsorbed-population arrays.
#include <cstdio>
#include <cstring>
#include <mutex>
#include <string>

#include "internal.cuh"

namespace mp {

namespace {

thread_local std::string g_last_error;

// one thread per node; a warp covers one 32-node word
__global__ void k_classify(const uint8_t* __restrict__ solid, int nx, int ny, int nz, int N, int W,
                           uint32_t* __restrict__ fluid_w, uint32_t* __restrict__ iface_w)
{
    int n = blockIdx.x * blockDim.x + threadIdx.x;
    bool fl = false, itf = false;
    if (n < N) {
        fl = solid[n] == 0;
        if (fl) {
            int x = n % nx, y = (n / nx) % ny, z = n / (nx * ny);
#pragma unroll
            for (int i = 1; i < kQ; ++i) {
                int xs = x + cx(i), ys = y + cy(i), zs = z + cz(i);
                xs = xs < 0 ? xs + nx : (xs >= nx ? xs - nx : xs);
                ys = ys < 0 ? ys + ny : (ys >= ny ? ys - ny : ys);
                zs = zs < 0 ? zs + nz : (zs >= nz ? zs - nz : zs);
                itf |= solid[xs + nx * (ys + ny * zs)] != 0;
            }
        }
    }
    unsigned bf = __ballot_sync(0xffffffffu, fl);
    unsigned bi = __ballot_sync(0xffffffffu, itf);
    int w = n >> 5;
    if ((threadIdx.x & 31) == 0 && w < W) {
        fluid_w[w] = bf;
        iface_w[w] = bi;
    }
}

// Exclusive prefixes of popc(iface_w) into ibase and of popc(fluid_w) into fbase, and the two
// totals: every block scans kScanWords words (four consecutive words a thread) and writes its
// totals, one block scans those, a third pass adds them (nothing to add with one block). One
// block walking the words a thread by a thread took 220 us of a 128^3 box, this takes about 8.
constexpr int kScanThreads = 256, kScanPer = 4, kScanWords = kScanThreads * kScanPer;

// inclusive scan of v over the block; s_w: one value per warp
__device__ __forceinline__ int block_scan(int v, int* s_w)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += t;
    }
    __syncthreads();
    if (lane == 31) s_w[warp] = v;
    __syncthreads();
    for (int k = 0; k < warp; ++k) v += s_w[k];
    return v;
}

__global__ void __launch_bounds__(kScanThreads)
    k_scan(const uint32_t* __restrict__ fluid_w, const uint32_t* __restrict__ iface_w, int W,
           int32_t* __restrict__ ibase, int32_t* __restrict__ fbase, int2* __restrict__ sums,
           long long* __restrict__ totals)
{
    __shared__ int s_w[kScanThreads / 32];
    const int w0 = blockIdx.x * kScanWords + threadIdx.x * kScanPer;
    int ci[kScanPer], cf[kScanPer], si = 0, sf = 0;
#pragma unroll
    for (int k = 0; k < kScanPer; ++k) {
        ci[k] = w0 + k < W ? __popc(iface_w[w0 + k]) : 0;
        cf[k] = w0 + k < W ? __popc(fluid_w[w0 + k]) : 0;
        si += ci[k];
        sf += cf[k];
    }
    const int ii = block_scan(si, s_w), ff = block_scan(sf, s_w);
    int ei = ii - si, ef = ff - sf;
#pragma unroll
    for (int k = 0; k < kScanPer; ++k) {
        if (w0 + k < W) {
            ibase[w0 + k] = ei;
            fbase[w0 + k] = ef;
        }
        ei += ci[k];
        ef += cf[k];
    }
    if (threadIdx.x == kScanThreads - 1) {
        sums[blockIdx.x] = make_int2(ii, ff);
        if (gridDim.x == 1) {
            totals[0] = ff;
            totals[1] = ii;
        }
    }
}

// one block: exclusive scan of the block totals in place, and the grand totals
__global__ void __launch_bounds__(kScanThreads) k_scan_sums(int2* __restrict__ sums, int nb, long long* __restrict__ totals)
{
    __shared__ int s_w[kScanThreads / 32];
    int bi = 0, bf = 0;  // totals of the blocks before this chunk
    for (int c0 = 0; c0 < nb; c0 += kScanThreads) {
        const int k = c0 + threadIdx.x;
        const int2 v = k < nb ? sums[k] : make_int2(0, 0);
        const int ii = block_scan(v.x, s_w), ff = block_scan(v.y, s_w);
        if (k < nb) sums[k] = make_int2(bi + ii - v.x, bf + ff - v.y);
        __shared__ int s_t[2];
        if (threadIdx.x == kScanThreads - 1) {
            s_t[0] = ii;
            s_t[1] = ff;
        }
        __syncthreads();
        bi += s_t[0];
        bf += s_t[1];
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        totals[0] = bf;
        totals[1] = bi;
    }
}

__global__ void __launch_bounds__(kScanThreads)
    k_scan_add(const int2* __restrict__ sums, int W, int32_t* __restrict__ ibase, int32_t* __restrict__ fbase)
{
    const int2 v = sums[blockIdx.x];
    for (int k = threadIdx.x; k < kScanWords; k += kScanThreads) {
        const int w = blockIdx.x * kScanWords + k;
        if (w < W) {
            ibase[w] += v.x;
            fbase[w] += v.y;
        }
    }
}

__global__ void k_list(const uint32_t* __restrict__ bits_w, const int32_t* __restrict__ base, int N,
                       int32_t* __restrict__ list)
{
    int n = blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= N) return;
    uint32_t bits = bits_w[n >> 5];
    int b = n & 31;
    if ((bits >> b) & 1u) list[base[n >> 5] + __popc(bits & ((1u << b) - 1u))] = n;
}

// Connected components by union-find. label[n] names a node of n's cluster with an index of at
// most n (its parent); a root names itself. Two roots are joined by lowering the larger one's
// label to the smaller with an atomic minimum, so labels only decrease and the root of a
// finished cluster is its smallest node, whatever the schedule. One pass over the links instead
// of sweeps until nothing changes (24 sweeps of 30-55 us and three waits for the host on a 128^3
// box of overlapping spheres).
__device__ __forceinline__ bool bit(const uint32_t* __restrict__ w, int n) { return (__ldg(w + (n >> 5)) >> (n & 31)) & 1u; }

__device__ __forceinline__ int uf_root(const int* label, int n)
{
    const volatile int* lab = label;
    int p = lab[n];
    while (p != n) {
        n = p;
        p = lab[n];
    }
    return n;
}

// joins the clusters of a and b; every round of the loop lowers a label
__device__ __forceinline__ void uf_join(int* label, int a, int b)
{
    while (true) {
        a = uf_root(label, a);
        b = uf_root(label, b);
        if (a == b) return;
        if (a < b) {
            const int t = a;
            a = b;
            b = t;
        }
        const int old = atomicMin(label + a, b);
        if (old == a) return;  // a was still a root
        a = old;               // another thread lowered it first: join that one with b
    }
}

// every fluid node starts with the first node of its run of fluid nodes in its row and word
__global__ void k_uf_init(const uint32_t* __restrict__ fluid_w, int N, int nx, int* __restrict__ label)
{
    const int n = blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= N) return;
    const uint32_t bits = __ldg(fluid_w + (n >> 5));
    const int b = n & 31;
    if (!((bits >> b) & 1u)) {
        label[n] = 0x7fffffff;
        return;
    }
    const uint32_t gaps = ~bits & ((1u << b) - 1u);
    const int run = n - b + (gaps ? 32 - __clz(gaps) : 0);
    label[n] = max(run, n - n % nx);
}

// joins every fluid node with its nine neighbours in links of one sign, leaving out those that
// the links of x-adjacent nodes imply (a row's adjacent fluid nodes are one cluster already)
__global__ void k_uf_join(const uint32_t* __restrict__ fluid_w, int nx, int ny, int nz, int N, int* label)
{
    const int n = blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= N || !bit(fluid_w, n)) return;
    const int x = n % nx, y = (n / nx) % ny, z = n / (nx * ny);
    const int row = n - x;
    const bool lo = x > 0, hi = x < nx - 1;
    const int xm = lo ? x - 1 : nx - 1, xp = hi ? x + 1 : 0;
    const bool left = bit(fluid_w, row + xm), right = bit(fluid_w, row + xp);
    if (left && (!lo || (n & 31) == 0)) uf_join(label, n, row + xm);
    const bool l = lo && left, r = hi && right;
    const int ym = y > 0 ? y - 1 : ny - 1, yp = y < ny - 1 ? y + 1 : 0, zm = z > 0 ? z - 1 : nz - 1;
    // rows (y-1, z) and (y, z-1): three links; (y-1, z-1) and (y+1, z-1): one
    const int rows[4] = {nx * (ym + ny * z), nx * (y + ny * zm), nx * (ym + ny * zm), nx * (yp + ny * zm)};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int o = rows[k];
        const bool m = bit(fluid_w, o + x);
        if (m && !(l && bit(fluid_w, o + x - 1))) uf_join(label, n, o + x);
        if (k < 2) {
            // x - 1: implied by n's link to (x) or by (x - 1)'s own where adjacent; x + 1 likewise
            if (!(lo && (m || l)) && bit(fluid_w, o + xm)) uf_join(label, n, o + xm);
            if (!(hi && (m || r)) && bit(fluid_w, o + xp)) uf_join(label, n, o + xp);
        }
    }
}

// label[n] = root, and the size of every cluster at its root: the nodes of a block that share
// the root of its first fluid node are added at once, the others warp by warp
__global__ void __launch_bounds__(256) k_cc_count(const uint32_t* __restrict__ fluid_w, int N, int* __restrict__ label,
                                                  int* __restrict__ count)
{
    __shared__ int s_first, s_root;
    const int n = blockIdx.x * 256 + threadIdx.x;
    const bool fl = n < N && bit(fluid_w, n);
    if (threadIdx.x == 0) s_first = 256;
    __syncthreads();
    int root = -1;
    if (fl) {
        root = uf_root(label, n);
        label[n] = root;
        atomicMin(&s_first, (int)threadIdx.x);
    }
    __syncthreads();
    if ((int)threadIdx.x == s_first) s_root = root;
    __syncthreads();
    const bool same = fl && root == s_root;
    const int c = __syncthreads_count(same);
    if (c > 0 && threadIdx.x == 0) atomicAdd(count + s_root, c);
    const unsigned rest = __ballot_sync(0xffffffffu, fl && !same);
    if (fl && !same) {
        const unsigned peers = __match_any_sync(rest, root);
        if ((int)(threadIdx.x & 31) == __ffs(peers) - 1) atomicAdd(count + root, __popc(peers));
    }
}

// key = size << 32 | (0xffffffff - root): the maximum is the largest cluster, ties to the
// smallest root index
__global__ void k_cc_best(const int* __restrict__ count, int N, unsigned long long* __restrict__ best)
{
    int n = blockIdx.x * blockDim.x + threadIdx.x;
    unsigned long long key = 0ull;
    if (n < N && count[n] > 0) key = ((unsigned long long)count[n] << 32) | (0xffffffffull - (unsigned)n);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        unsigned long long v = __shfl_xor_sync(0xffffffffu, key, o);
        key = v > key ? v : key;
    }
    if ((threadIdx.x & 31) == 0 && key) atomicMax(best, key);
}

__global__ void k_cc_mark(const uint32_t* __restrict__ fluid_w, int N, int W, const int* __restrict__ label,
                          const unsigned long long* __restrict__ best, uint32_t* __restrict__ cluster_w)
{
    int n = blockIdx.x * blockDim.x + threadIdx.x;
    const int root = (int)(0xffffffffull - (*best & 0xffffffffull));
    bool in = n < N && ((fluid_w[n >> 5] >> (n & 31)) & 1u) && label[n] == root;
    unsigned b = __ballot_sync(0xffffffffu, in);
    if ((threadIdx.x & 31) == 0 && (n >> 5) < W) cluster_w[n >> 5] = b;
}

// node classes as bytes: 0 solid, 1 fluid, 2 interfacial, plus 4 in the largest cluster; four
// nodes a thread
__global__ void k_class_bytes(const uint32_t* __restrict__ fluid_w, const uint32_t* __restrict__ iface_w,
                              const uint32_t* __restrict__ cluster_w, int N, uint8_t* __restrict__ cls, int vec)
{
    const int n = 4 * (blockIdx.x * blockDim.x + threadIdx.x);
    if (n >= N) return;
    const int w = n >> 5, b = n & 31;
    const uint32_t f = fluid_w[w] >> b, i = iface_w[w] >> b, c = cluster_w[w] >> b;
    uint32_t v = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) v |= (((f >> k) & 1u) + ((i >> k) & 1u) + 4u * ((c >> k) & 1u)) << (8 * k);
    if (vec && n + 3 < N) {
        *reinterpret_cast<uint32_t*>(cls + n) = v;
    } else {
        for (int k = 0; k < 4 && n + k < N; ++k) cls[n + k] = (uint8_t)(v >> (8 * k));
    }
}

template <typename T>
int dev_alloc(T** p, size_t count, cudaStream_t s, bool stream_ordered)
{
    cudaError_t e = stream_ordered ? pool_malloc((void**)p, count * sizeof(T), s)
                                   : cudaMalloc((void**)p, count * sizeof(T));
    if (e != cudaSuccess) {
        *p = nullptr;
        (void)cudaGetLastError();
        set_error(std::string("device allocation failed: ") + cudaGetErrorString(e));
        return MP_ENOMEM;
    }
    return MP_OK;
}

template <typename T>
void dev_free(T*& p, cudaStream_t s, bool stream_ordered)
{
    if (p) {
        if (stream_ordered)
            cudaFreeAsync(p, s);
        else
            cudaFree(p);
    }
    p = nullptr;
}

}  // namespace

// Stream-ordered scratch of the calls that allocate and free within themselves (lb_steady,
// mp_classify). The device's default pool gives everything back to the system at every
// synchronisation, so that each call maps its memory again; a pool of the library keeps up to
// kPoolKeep bytes mapped between calls instead. One pool per device and context (a new context
// after cudaDeviceReset gets a new one). Pools are safe across threads and streams;
// mp_release_cached gives the kept memory back.
namespace {
constexpr unsigned long long kPoolKeep = 256ull << 20;
constexpr int kPoolDevices = 64, kPoolContexts = 4;  // further contexts of a device use its default pool
struct PoolSlot {
    cudaMemPool_t pool = nullptr;
    unsigned long long ctx = 0;
};
std::mutex g_pool_mu;
PoolSlot g_pool[kPoolDevices][kPoolContexts];

cudaMemPool_t library_pool()
{
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kPoolDevices) return nullptr;
    const unsigned long long ctx = current_ctx_id();
    if (ctx == 0) return nullptr;
    std::lock_guard<std::mutex> lock(g_pool_mu);
    for (PoolSlot& slot : g_pool[dev]) {
        if (slot.pool && slot.ctx == ctx) return slot.pool;
        if (slot.pool) continue;
        cudaMemPoolProps props = {};
        props.allocType = cudaMemAllocationTypePinned;
        props.location.type = cudaMemLocationTypeDevice;
        props.location.id = dev;
        cudaMemPool_t p = nullptr;
        unsigned long long keep = kPoolKeep;
        if (cudaMemPoolCreate(&p, &props) != cudaSuccess) {
            (void)cudaGetLastError();
            return nullptr;
        }
        if (cudaMemPoolSetAttribute(p, cudaMemPoolAttrReleaseThreshold, &keep) != cudaSuccess) {
            (void)cudaGetLastError();
            cudaMemPoolDestroy(p);
            return nullptr;
        }
        slot.pool = p;
        slot.ctx = ctx;
        return p;
    }
    return nullptr;
}
}  // namespace

// The driver's context queries are resolved through the runtime, so the library needs no link
// to libcuda.
unsigned long long current_ctx_id()
{
    typedef int (*GetCurrentFn)(void**);
    typedef int (*GetIdFn)(void*, unsigned long long*);
    struct Fns {
        GetCurrentFn current = nullptr;
        GetIdFn id = nullptr;
    };
    static const Fns fns = [] {
        Fns f;
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            f.current = reinterpret_cast<GetCurrentFn>(p);
        p = nullptr;
        if (cudaGetDriverEntryPointByVersion("cuCtxGetId", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            f.id = reinterpret_cast<GetIdFn>(p);
        return f;
    }();
    void* ctx = nullptr;
    unsigned long long id = 0;
    if (!fns.current || !fns.id || fns.current(&ctx) != 0 || !ctx || fns.id(ctx, &id) != 0) return 0;
    return id;
}

cudaError_t pool_malloc(void** p, size_t bytes, cudaStream_t s)
{
    cudaMemPool_t pool = library_pool();
    return pool ? cudaMallocFromPoolAsync(p, bytes, pool, s) : cudaMallocAsync(p, bytes, s);
}

void pool_trim()
{
    if (cudaMemPool_t pool = library_pool()) {
        cudaDeviceSynchronize();
        cudaMemPoolTrimTo(pool, 0);
    }
    (void)cudaGetLastError();
}

void set_error(const std::string& msg) { g_last_error = msg; }
void clear_error() { g_last_error.clear(); }
const char* last_error_text() { return g_last_error.c_str(); }

int cuda_fail(cudaError_t e, const char* what)
{
    set_error(std::string("CUDA error in ") + what + ": " + cudaGetErrorString(e));
    if (e == cudaErrorMemoryAllocation) return MP_ENOMEM;
    return MP_ECUDA;
}

void free_geometry(Geometry* g, cudaStream_t s, bool so)
{
    dev_free(g->cluster, s, so);
    dev_free(g->fluid, s, so);
    dev_free(g->iface, s, so);
    dev_free(g->ibase, s, so);
    dev_free(g->ilist, s, so);
    dev_free(g->fbase, s, so);
    dev_free(g->flist, s, so);
}

int build_cluster(Geometry* G, cudaStream_t s, bool so, bool want_count)
{
    int* label = nullptr;
    int* count = nullptr;
    unsigned long long* best = nullptr;
    int rc;
    if ((rc = dev_alloc(&G->cluster, G->W, s, so)) || (rc = dev_alloc(&label, G->N, s, so)) ||
        (rc = dev_alloc(&count, G->N, s, so)) || (rc = dev_alloc(&best, 1, s, so))) {
        dev_free(label, s, so);
        dev_free(count, s, so);
        dev_free(best, s, so);
        return rc;
    }
    const int threads = 256, blocks = (G->N + threads - 1) / threads;
    const int wblocks = (int)(((long long)G->W * 32 + threads - 1) / threads);
    k_uf_init<<<blocks, threads, 0, s>>>(G->fluid, G->N, G->nx, label);
    k_uf_join<<<blocks, threads, 0, s>>>(G->fluid, G->nx, G->ny, G->nz, G->N, label);
    cudaError_t e = cudaMemsetAsync(count, 0, sizeof(int) * (size_t)G->N, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(best, 0, sizeof(unsigned long long), s);
    if (e == cudaSuccess) {
        k_cc_count<<<blocks, 256, 0, s>>>(G->fluid, G->N, label, count);
        k_cc_best<<<blocks, threads, 0, s>>>(count, G->N, best);
        k_cc_mark<<<wblocks, threads, 0, s>>>(G->fluid, G->N, G->W, label, best, G->cluster);
        e = cudaGetLastError();
    }
    unsigned long long h_best = 0;
    if (want_count && e == cudaSuccess) {
        e = cudaMemcpyAsync(&h_best, best, sizeof(h_best), cudaMemcpyDeviceToHost, s);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    }
    dev_free(label, s, so);
    dev_free(count, s, so);
    dev_free(best, s, so);
    if (e != cudaSuccess) return cuda_fail(e, "connected clusters");
    G->n_cluster = (int64_t)(h_best >> 32);
    return MP_OK;
}

int build_geometry(const mp_geometry* g, cudaStream_t s, bool so, bool want_list, Geometry* out)
{
    if (!g || !g->solid) {
        set_error("geometry or its solid mask is NULL");
        return MP_EINVAL;
    }
    if (g->nx < 3 || g->ny < 3 || g->nz < 3) {
        set_error("every lattice dimension must be >= 3");
        return MP_EINVAL;
    }
    long long N = (long long)g->nx * g->ny * g->nz;
    // per-node launches round the node count up to whole 256-thread blocks in int
    // arithmetic, and node indices stay below 2^31
    if (N > (1LL << 31) - 256) {
        set_error("lattice too large: nx*ny*nz must be at most 2^31 - 256");
        return MP_EINVAL;
    }
    if (g->location != MP_HOST && g->location != MP_DEVICE) {
        set_error("geometry location must be MP_HOST or MP_DEVICE");
        return MP_EINVAL;
    }
    Geometry G;
    G.nx = g->nx;
    G.ny = g->ny;
    G.nz = g->nz;
    G.N = (int)N;
    G.W = (int)((N + 31) / 32);
    int rc;
    uint8_t* solid_d = nullptr;
    long long* totals = nullptr;
    int2* sums = nullptr;
    const int nb = (G.W + kScanWords - 1) / kScanWords;
    if ((rc = dev_alloc(&G.fluid, G.W, s, so)) || (rc = dev_alloc(&G.iface, G.W, s, so)) ||
        (rc = dev_alloc(&G.ibase, G.W, s, so)) || (rc = dev_alloc(&G.fbase, G.W, s, so)) ||
        (rc = dev_alloc(&totals, 2, s, so)) || (rc = dev_alloc(&sums, nb, s, so))) {
        free_geometry(&G, s, so);
        dev_free(totals, s, so);
        return rc;
    }
    const uint8_t* solid = g->solid;
    if (g->location == MP_HOST) {
        if ((rc = dev_alloc(&solid_d, (size_t)N, s, so))) {
            free_geometry(&G, s, so);
            dev_free(totals, s, so);
            dev_free(sums, s, so);
            return rc;
        }
        cudaError_t e = cudaMemcpyAsync(solid_d, g->solid, (size_t)N, cudaMemcpyHostToDevice, s);
        if (e != cudaSuccess) {
            free_geometry(&G, s, so);
            dev_free(totals, s, so);
            dev_free(sums, s, so);
            dev_free(solid_d, s, so);
            return cuda_fail(e, "cudaMemcpyAsync(solid)");
        }
        solid = solid_d;
    }
    int threads = 256;
    int blocks = (int)(((long long)G.W * 32 + threads - 1) / threads);
    k_classify<<<blocks, threads, 0, s>>>(solid, G.nx, G.ny, G.nz, G.N, G.W, G.fluid, G.iface);
    k_scan<<<nb, kScanThreads, 0, s>>>(G.fluid, G.iface, G.W, G.ibase, G.fbase, sums, totals);
    if (nb > 1) {
        k_scan_sums<<<1, kScanThreads, 0, s>>>(sums, nb, totals);
        k_scan_add<<<nb, kScanThreads, 0, s>>>(sums, G.W, G.ibase, G.fbase);
    }
    long long h_tot[2] = {0, 0};
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaMemcpyAsync(h_tot, totals, sizeof(h_tot), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    dev_free(solid_d, s, so);
    dev_free(totals, s, so);
    dev_free(sums, s, so);
    if (e != cudaSuccess) {
        free_geometry(&G, s, so);
        return cuda_fail(e, "geometry classification");
    }
    G.n_fluid = h_tot[0];
    G.n_iface = h_tot[1];
    if (want_list) {
        if ((G.n_iface > 0 && (rc = dev_alloc(&G.ilist, (size_t)G.n_iface, s, so))) ||
            (G.n_fluid > 0 && (rc = dev_alloc(&G.flist, (size_t)G.n_fluid, s, so)))) {
            free_geometry(&G, s, so);
            return rc;
        }
        if (G.n_iface > 0) k_list<<<(G.N + 255) / 256, 256, 0, s>>>(G.iface, G.ibase, G.N, G.ilist);
        if (G.n_fluid > 0) k_list<<<(G.N + 255) / 256, 256, 0, s>>>(G.fluid, G.fbase, G.N, G.flist);
        e = cudaGetLastError();
        if (e != cudaSuccess) {
            free_geometry(&G, s, so);
            return cuda_fail(e, "node lists");
        }
    }
    *out = G;
    return MP_OK;
}

}  // namespace mp

namespace {

// classes to host memory (cls) or device memory (cls_dev); the counts are written when given
int classify(const mp_geometry* g, uint8_t* cls, uint8_t* cls_dev, int64_t* n_fluid, int64_t* n_interface,
             int64_t* n_cluster, cudaStream_t s)
{
    using namespace mp;
    Geometry G;
    uint8_t* tmp = nullptr;
    int rc = build_geometry(g, s, true, false, &G);
    if (rc == MP_OK) rc = build_cluster(&G, s, true, n_cluster != nullptr);
    cudaError_t e = cudaSuccess;
    if (rc == MP_OK && !cls_dev) {
        e = pool_malloc((void**)&tmp, (size_t)G.N, s);
        if (e != cudaSuccess) {
            (void)cudaGetLastError();
            tmp = nullptr;
            set_error(std::string("device allocation failed: ") + cudaGetErrorString(e));
            rc = MP_ENOMEM;
        }
    }
    if (rc == MP_OK) {
        uint8_t* out = cls_dev ? cls_dev : tmp;
        const int quads = (int)(((long long)G.N + 3) / 4);
        k_class_bytes<<<(quads + 255) / 256, 256, 0, s>>>(G.fluid, G.iface, G.cluster, G.N, out,
                                                          ((uintptr_t)out & 3) == 0);
        e = cudaGetLastError();
        if (e == cudaSuccess && !cls_dev) {
            e = cudaMemcpyAsync(cls, tmp, (size_t)G.N, cudaMemcpyDeviceToHost, s);
            if (e == cudaSuccess) e = cudaStreamSynchronize(s);
        }
        if (n_fluid) *n_fluid = G.n_fluid;
        if (n_interface) *n_interface = G.n_iface;
        if (n_cluster) *n_cluster = G.n_cluster;
        if (e != cudaSuccess) rc = cuda_fail(e, "mp_classify");
    }
    if (tmp) cudaFreeAsync(tmp, s);
    free_geometry(&G, s, true);
    if (rc != MP_OK) cudaStreamSynchronize(s);
    return rc;
}

}  // namespace

extern "C" int mp_classify(const mp_geometry* g, uint8_t* cls, int64_t* n_fluid, int64_t* n_interface,
                           int64_t* n_cluster, void* stream)
{
    mp::clear_error();
    if (!cls) {
        mp::set_error("mp_classify: cls is NULL");
        return MP_EINVAL;
    }
    return classify(g, cls, nullptr, n_fluid, n_interface, n_cluster, (cudaStream_t)stream);
}

extern "C" int mp_classify_device(const mp_geometry* g, uint8_t* cls, int64_t* n_fluid, int64_t* n_interface,
                                  int64_t* n_cluster, void* stream)
{
    mp::clear_error();
    if (!cls) {
        mp::set_error("mp_classify_device: cls is NULL");
        return MP_EINVAL;
    }
    return classify(g, nullptr, cls, n_fluid, n_interface, n_cluster, (cudaStream_t)stream);
}

extern "C" void mp_release_cached(void) { mp::pool_trim(); }
