// Many time steps of a small lattice in one launch, with the state resident in
// the shared memory of one thread-block cluster.
//
// A step of a lattice of a few thousand cells moves less than a megabyte: a
// launch per step costs far more than the step, even replayed from a graph.
// Here a cluster of up to 16 blocks (one per SM) holds both population buffers in its
// shared memory; block r owns the cells [r * chunk, (r + 1) * chunk) and a
// thread up to kCells of them. Every thread resolves the pull sources of its
// cells once, as shared-memory addresses within the cluster (own block or a
// neighbour's, with the periodic wrap, walls and obstacles folded in), so a
// step is q loads, the collision and q local stores per cell, then one cluster
// barrier. The collision is the one of the per-cell kernels: the same bits.
#include "k_step.cuh"

namespace hlbm {

namespace {

constexpr int kBlocks = 16;       // blocks of the cluster, one per SM (8 measured up to 30 % slower, 4 up to 2x)
constexpr int kMaxThreads = 512;  // per block

__device__ __forceinline__ unsigned cluster_rank() {
    unsigned r;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ unsigned map_rank(unsigned a, unsigned rank) {
    unsigned r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
    return r;
}
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// Population at a shared address of the cluster, in the arithmetic type.
template <class S>
__device__ __forceinline__ float ld_cluster(unsigned a) {
    if constexpr (S::kind == 1) {
        float v;
        asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(a) : "memory");
        return v;
    } else {
        unsigned short h;
        asm volatile("ld.shared::cluster.u16 %0, [%1];" : "=h"(h) : "r"(a) : "memory");
        if constexpr (S::kind == 2) return __half2float(__ushort_as_half(h));
        else return __bfloat162float(__ushort_as_bfloat16(h));
    }
}

template <int Q, class S, int FORM, int CELLS>
__global__ void __launch_bounds__(kMaxThreads, 1)
k_resident(typename S::T* f, const float* __restrict__ varpi, Geometry g, Phys<float> ph, float s, float inv_s,
           const float* __restrict__ varpi3, const unsigned* __restrict__ links, int chunk, int nsteps) {
    using T = typename S::T;
    extern __shared__ __align__(16) unsigned char resident_smem[];
    T* const sm = reinterpret_cast<T*>(resident_smem);
    const int N = (int)g.N, base = (int)cluster_rank() * chunk;
    const unsigned sm0 = (unsigned)__cvta_generic_to_shared(sm);
    const int buffer = Q * chunk;  // values of one population buffer of a block

    unsigned src[CELLS][Q];
    float vp[CELLS][FORM == FORM_ANISO ? 3 : 1];
    bool live[CELLS];
#pragma unroll
    for (int k = 0; k < CELLS; ++k) {
        const int l = (int)threadIdx.x + k * (int)blockDim.x, cell = base + l;
        live[k] = l < chunk && cell < N;
        if (!live[k]) continue;
        const int x = cell % g.nx, yz = cell / g.nx, y = yz % g.ny, z = yz / g.ny;
        const unsigned lm = links ? __ldg(links + cell) : 0u;
        live[k] = !(lm & kSolidBit);  // solid cells are neither updated nor read
        if (!live[k]) continue;
        const Nbr<int> nb(g, x, y, z, lm);
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            sm[i * chunk + l] = f[(size_t)i * N + cell];
            const bool wall = nb.template beyond_wall<Q>(i, -1);
            const int j = wall ? opp<Q>(i) : i, from = wall ? cell : cell + nb.template offset<Q>(i, -1);
            const int owner = from / chunk;
            src[k][i] = map_rank(sm0 + (unsigned)(j * chunk + (from - owner * chunk)) * (unsigned)sizeof(T), (unsigned)owner);
        }
        if constexpr (FORM == FORM_ANISO) {
#pragma unroll
            for (int a = 0; a < 3; ++a) vp[k][a] = __ldg(varpi3 + (size_t)a * N + cell);
        } else {
            vp[k][0] = __ldg(varpi + cell);
        }
    }
    cluster_sync();
    for (int n = 0; n < nsteps; ++n) {
        const unsigned from = (n & 1) ? (unsigned)buffer * (unsigned)sizeof(T) : 0u;
        T* const to = sm + ((n & 1) ? 0 : buffer);
#pragma unroll
        for (int k = 0; k < CELLS; ++k) {
            if (!live[k]) continue;
            float d[Q];
#pragma unroll
            for (int i = 0; i < Q; ++i) d[i] = ld_cluster<S>(src[k][i] + from);
            const WriteBack<float> out{d};
            if constexpr (FORM == FORM_ANISO) collide_aniso<Q, float, S::scaled>(d, vp[k][0], vp[k][1], vp[k][2], ph, s, inv_s, out);
            else if constexpr (FORM == FORM_DRAG) collide_drag<Q, float, S::scaled>(d, vp[k][0], ph, s, inv_s, out);
            else collide<Q, float, S::scaled, FORM == FORM_SHIFT_FX>(d, vp[k][0], ph, s, inv_s, out);
            const int l = (int)threadIdx.x + k * (int)blockDim.x;
#pragma unroll
            for (int i = 0; i < Q; ++i) S::store_raw(to, i * chunk + l, d[i]);
        }
        cluster_sync();
    }
    const T* const last = sm + ((nsteps & 1) ? buffer : 0);
#pragma unroll
    for (int k = 0; k < CELLS; ++k) {
        const int l = (int)threadIdx.x + k * (int)blockDim.x;
        if (!live[k]) continue;
#pragma unroll
        for (int i = 0; i < Q; ++i) f[(size_t)i * N + base + l] = last[i * chunk + l];
    }
}

struct ResidentPlan {
    int threads, cells, chunk;  // threads per block, cells per thread, cells per block
};
ResidentPlan plan(const LaunchCtx& c) {
    const int n = c.nx * c.ny * c.nz;
    ResidentPlan p{0, 1, (n + kBlocks - 1) / kBlocks};
    if (p.chunk > kMaxThreads) p.cells = 2;
    p.threads = ((p.chunk + p.cells - 1) / p.cells + 31) / 32 * 32;
    return p;
}

template <int Q, class S, int FORM, int CELLS>
cudaError_t resident_impl(const LaunchCtx& c, const ResidentPlan& p, void* f, const float* varpi, int nsteps) {
    using T = typename S::T;
    const auto kern = k_resident<Q, S, FORM, CELLS>;
    const int bytes = 2 * Q * p.chunk * (int)sizeof(T);
    // The limit is the kernel's largest size, not this launch's: several threads may launch it.
    constexpr int kMaxBytes = 2 * Q * CELLS * kMaxThreads * (int)sizeof(T);
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxBytes);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    const Geometry g{c.nx, c.ny, c.nz, c.wall[0], c.wall[1], c.wall[2], (size_t)c.nx * c.ny * c.nz};
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(kBlocks);
    cfg.blockDim = dim3(p.threads);
    cfg.dynamicSmemBytes = bytes;
    cfg.stream = c.stream;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = kBlocks;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, static_cast<T*>(f), varpi, g, make_phys<float, Q>(c.tau, c.F), float(c.scale),
                              float(1.0 / c.scale), c.varpi3, c.links, p.chunk, nsteps);
}

template <int Q, class S, int FORM>
cudaError_t resident_cells(const LaunchCtx& c, const ResidentPlan& p, void* f, const float* varpi, int nsteps) {
    if constexpr (Q == 9)
        if (p.cells == 2) return resident_impl<Q, S, FORM, 2>(c, p, f, varpi, nsteps);
    return resident_impl<Q, S, FORM, 1>(c, p, f, varpi, nsteps);
}
template <int Q, class S>
cudaError_t resident_form(const LaunchCtx& c, const ResidentPlan& p, void* f, const float* varpi, int nsteps) {
    switch (step_form(c, Q)) {
        case FORM_SHIFT_FX: return resident_cells<Q, S, FORM_SHIFT_FX>(c, p, f, varpi, nsteps);
        case FORM_SHIFT: return resident_cells<Q, S, FORM_SHIFT>(c, p, f, varpi, nsteps);
        case FORM_DRAG: return resident_cells<Q, S, FORM_DRAG>(c, p, f, varpi, nsteps);
        default: return resident_cells<Q, S, FORM_ANISO>(c, p, f, varpi, nsteps);
    }
}
template <class S>
cudaError_t resident_q(const LaunchCtx& c, const ResidentPlan& p, void* f, const float* varpi, int nsteps) {
    return c.q == 9 ? resident_form<9, S>(c, p, f, varpi, nsteps) : resident_form<19, S>(c, p, f, varpi, nsteps);
}

// Largest lattice per velocity set: D2Q9 two cells per thread, D3Q19 one. Measured,
// us per step, resident vs one launch per step replayed from a graph (FP32): D2Q9
// 64x32 0.51 vs 1.80, 96x64 0.61 vs 2.05, 128x96 0.96 vs 2.05; D3Q19 12^3 0.78 vs
// 2.31, 16^3 (drag, walls) 1.08 vs 2.82, 20^3 1.72 vs 2.56; at two cells per
// thread D3Q19 loses (24^3 2.31 vs 2.56, 32x32x16 2.81 vs 2.31): sixteen SMs then
// take longer than the whole chip and a launch.
size_t resident_cells_max(int q) { return (size_t)kBlocks * kMaxThreads * (q == 9 ? 2 : 1); }

// Can the current context run the largest cluster (16 blocks is beyond the portable size: it
// needs sixteen free SMs behind one cluster scheduler)?
int ask_cluster() {
    const auto kern = k_resident<19, StoreF32, FORM_SHIFT, 1>;
    const int bytes = 2 * 19 * kMaxThreads * (int)sizeof(float);
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(kBlocks);
    cfg.blockDim = dim3(kMaxThreads);
    cfg.dynamicSmemBytes = bytes;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = kBlocks;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int n = 0;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveClusters(&n, kern, &cfg);
    if (e == cudaSuccess) return n >= 1;
    (void)cudaGetLastError();
    return -1;
}
ContextFact g_cluster;

}  // namespace

bool resident_applies(const LaunchCtx& c) {
    return c.variant == 0 && c.storage != 0 && (size_t)c.nx * c.ny * c.nz <= resident_cells_max(c.q) && g_cluster.get(ask_cluster);
}

cudaError_t launch_resident(const LaunchCtx& c, void* f, const float* varpi, int nsteps) {
    const ResidentPlan p = plan(c);
    switch (c.storage) {
        case 1: return resident_q<StoreF32>(c, p, f, varpi, nsteps);
        case 2: return resident_q<StoreF16>(c, p, f, varpi, nsteps);
        case 3: return resident_q<StoreBF16>(c, p, f, varpi, nsteps);
    }
    return cudaErrorInvalidValue;
}

}  // namespace hlbm
