// Observables and state I/O: moments, population conversion, input validation.
#include "dispatch.cuh"

namespace hlbm {

// ---------------------------------------------------------------------------
// Moments (Def. moments of the streamed populations, half-force velocity).
// ---------------------------------------------------------------------------
// LAY: the state's layout with 32-bit indices, or -1 (any layout, 64-bit indices).
template <int Q, class S, bool WALLS, class Out, int LAY>
__global__ void __launch_bounds__(256)
k_moments(const typename S::T* f, int lay, Geometry g, Phys<typename S::C> ph, typename S::C inv_s,
          Out* rho, Out* u, const float* varpi, int drag, const unsigned* links) {
    using C = typename S::C;
    using I = typename std::conditional<LAY >= 0, int, long long>::type;
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y * blockDim.y + threadIdx.y;
    const int z = blockIdx.z;
    if (x >= g.nx || y >= g.ny) return;
    const I cell = (I)x + (I)g.nx * ((I)y + (I)g.ny * (I)z);
    const unsigned lm = links ? links[cell] : 0u;
    if (lm & kSolidBit) {  // resolved obstacle: at rest
        if (rho) rho[cell] = Out(1);
        if (u) u[cell] = u[g.N + cell] = u[2 * g.N + cell] = Out(0);
        return;
    }
    const Nbr<I> nb(g, x, y, z, lm);
    C d[Q];
#pragma unroll
    for (int i = 0; i < Q; ++i) d[i] = S::load(f, gather_index<Q, WALLS>(g, nb, cell, i, LAY >= 0 ? LAY : lay), inv_s);
    C drho, jx, jy, jz;
    moments<Q, C>(d, drho, jx, jy, jz);
    const C r = C(1) + drho;
    if (rho) rho[cell] = Out(r);
    if (u) {
        C ux, uy, uz;
        velocity_form<C>(jx, jy, jz, r, drag ? C(varpi[cell]) : C(1), drag, ph, ux, uy, uz);
        u[cell] = Out(ux);
        u[g.N + cell] = Out(uy);
        u[2 * g.N + cell] = Out(uz);
    }
}

template <int Q, class S, bool WALLS>
static cudaError_t moments_impl(const LaunchCtx& c, int lay, const void* f, void* rho, void* u, int f64) {
    using C = typename S::C;
    const Geometry g = geom(c);
    const dim3 blk = row_block(c.nx, c.ny);
    const dim3 grd((c.nx + blk.x - 1) / blk.x, (c.ny + blk.y - 1) / blk.y, c.nz);
    const auto* a = static_cast<const typename S::T*>(f);
    with_layout((size_t)Q * g.N, lay, [&]<int LAY>() {
        if (f64)
            k_moments<Q, S, WALLS, double, LAY><<<grd, blk, 0, c.stream>>>(a, lay, g, phys<C, Q>(c), C(1.0 / c.scale),
                                                                           (double*)rho, (double*)u, c.varpi, c.drag, c.links);
        else
            k_moments<Q, S, WALLS, float, LAY><<<grd, blk, 0, c.stream>>>(a, lay, g, phys<C, Q>(c), C(1.0 / c.scale),
                                                                          (float*)rho, (float*)u, c.varpi, c.drag, c.links);
    });
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// State conversion (natural FP64 full populations <-> stored deviations).
// ---------------------------------------------------------------------------
template <int Q, class S, bool WALLS>
__global__ void __launch_bounds__(256)
k_write_state(const double* fnat, int uniform, int lay, Geometry g, typename S::C s, typename S::T* f,
              const unsigned* links) {
    using C = typename S::C;
    using L = Lat<Q>;
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y * blockDim.y + threadIdx.y;
    const int z = blockIdx.z;
    if (x >= g.nx || y >= g.ny) return;
    const long long cell = (long long)x + (long long)g.nx * ((long long)y + (long long)g.ny * (long long)z);
    const unsigned lm = links ? links[cell] : 0u;
    if (lm & kSolidBit) return;  // solid cells hold no state (their slots may belong to neighbours)
    const Nbr<long long> nb(g, x, y, z, lm);
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        const double fi = uniform ? fnat[i] : fnat[(size_t)i * g.N + cell];
        S::store(f, natural_index<Q, WALLS>(g, nb, cell, i, lay), C(fi - L::w(i)), s);
    }
}

// Rest populations (deviation 0) into the slots of the solid cells, which are theirs alone in every
// layout: no step reads or writes them, so they keep what this kernel leaves.
template <int Q, class S>
__global__ void __launch_bounds__(256) k_rest_solid(typename S::T* f, Geometry g, const unsigned* links) {
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y * blockDim.y + threadIdx.y;
    const int z = blockIdx.z;
    if (x >= g.nx || y >= g.ny) return;
    const size_t cell = (size_t)x + (size_t)g.nx * ((size_t)y + (size_t)g.ny * (size_t)z);
    if (!(links[cell] & kSolidBit)) return;
#pragma unroll
    for (int i = 0; i < Q; ++i) f[(size_t)i * g.N + cell] = typename S::T(0.0f);
}

// float -> double, exactly, on the integer pipe: a conversion instruction runs on the
// FP64 pipe, which the addition of the weight below already keeps busy (two lanes
// per clock and SM). Zero and normal values; the others take the instruction.
__device__ __forceinline__ double widen(float v) {
    const unsigned b = __float_as_uint(v);
    if ((b << 1) - 0x01000000u < 0xfe000000u)  // exponent 1..254
        return __hiloint2double((int)((b & 0x80000000u) | (((b & 0x7fffffffu) >> 3) + 0x38000000u)), (int)(b << 29));
    if ((b << 1) == 0u) return __hiloint2double((int)b, 0);
    return (double)v;
}
__device__ __forceinline__ double widen(double v) { return v; }

// Populations as FP64 full values: 8 q bytes written per cell next to the state's
// read, and q FP64 additions per cell, which bound it. Measured, a conversion
// instruction per value vs widen(): 256^3 FP32 1178 vs 763 us (3.8 GB), in-place BF16
// 192^3 503 vs 314 us.
template <int Q, class S, bool WALLS, int LAY>
__global__ void __launch_bounds__(256)
k_read_state(const typename S::T* __restrict__ f, int lay, Geometry g, typename S::C inv_s, double* __restrict__ fnat,
             const unsigned* __restrict__ links) {
    using L = Lat<Q>;
    using I = typename std::conditional<LAY >= 0, int, long long>::type;
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y * blockDim.y + threadIdx.y;
    const int z = blockIdx.z;
    if (x >= g.nx || y >= g.ny) return;
    const I cell = (I)x + (I)g.nx * ((I)y + (I)g.ny * (I)z), N = (I)g.N;
    const unsigned lm = links ? links[cell] : 0u;
    if (lm & kSolidBit) {  // solid cells read as the rest state
#pragma unroll
        for (int i = 0; i < Q; ++i) fnat[(I)i * N + cell] = L::w(i);
        return;
    }
    const Nbr<I> nb(g, x, y, z, lm);
#pragma unroll
    for (int i = 0; i < Q; ++i)
        fnat[(I)i * N + cell] =
            L::w(i) + widen(S::load(f, natural_index<Q, WALLS>(g, nb, cell, i, LAY >= 0 ? LAY : lay), inv_s));
}

// The same state as k_write_state with uniform = 1 (every cell holds fnat[i]),
// for kFillZ consecutive z planes per thread: the deviation of each direction
// is formed once per thread (in double, as k_write_state forms it, so the bits
// are the same), and the per-cell work is only the index and the store. GB300's
// FP64 rate is a small fraction of its FP32 rate, and the per-cell double
// subtract and conversion had limited the initial write to about 1.2 TB/s.
constexpr int kFillZ = 8;

template <int Q, class S, bool WALLS>
__global__ void __launch_bounds__(256)
k_fill_state(const double* fnat, int lay, Geometry g, typename S::C s, typename S::T* f, const unsigned* links) {
    using C = typename S::C;
    using L = Lat<Q>;
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y * blockDim.y + threadIdx.y;
    if (x >= g.nx || y >= g.ny) return;
    C v[Q];
#pragma unroll
    for (int i = 0; i < Q; ++i) v[i] = C(fnat[i] - L::w(i));
    const int z0 = blockIdx.z * kFillZ;
    const int z1 = z0 + kFillZ < g.nz ? z0 + kFillZ : g.nz;
    for (int z = z0; z < z1; ++z) {
        const long long cell = (long long)x + (long long)g.nx * ((long long)y + (long long)g.ny * (long long)z);
        const unsigned lm = links ? links[cell] : 0u;
        if (lm & kSolidBit) continue;
        const Nbr<long long> nb(g, x, y, z, lm);
#pragma unroll
        for (int i = 0; i < Q; ++i) S::store(f, natural_index<Q, WALLS>(g, nb, cell, i, lay), v[i], s);
    }
}

template <int Q, class S, bool WALLS>
static cudaError_t write_impl(const LaunchCtx& c, int lay, const double* fnat, int uniform, void* f) {
    using C = typename S::C;
    const dim3 blk = row_block(c.nx, c.ny);
    if (uniform) {
        const dim3 grd((c.nx + blk.x - 1) / blk.x, (c.ny + blk.y - 1) / blk.y, (c.nz + kFillZ - 1) / kFillZ);
        k_fill_state<Q, S, WALLS><<<grd, blk, 0, c.stream>>>(fnat, lay, geom(c), C(c.scale),
                                                             static_cast<typename S::T*>(f), c.links);
        return cudaGetLastError();
    }
    const dim3 grd((c.nx + blk.x - 1) / blk.x, (c.ny + blk.y - 1) / blk.y, c.nz);
    k_write_state<Q, S, WALLS><<<grd, blk, 0, c.stream>>>(fnat, uniform, lay, geom(c), C(c.scale),
                                                          static_cast<typename S::T*>(f), c.links);
    return cudaGetLastError();
}

template <int Q, class S, bool WALLS>
static cudaError_t read_impl(const LaunchCtx& c, int lay, const void* f, double* fnat) {
    using C = typename S::C;
    const dim3 blk = row_block(c.nx, c.ny);
    const dim3 grd((c.nx + blk.x - 1) / blk.x, (c.ny + blk.y - 1) / blk.y, c.nz);
    with_layout((size_t)Q * c.nx * c.ny * c.nz, lay, [&]<int LAY>() {
        k_read_state<Q, S, WALLS, LAY><<<grd, blk, 0, c.stream>>>(static_cast<const typename S::T*>(f), lay, geom(c),
                                                                  C(1.0 / c.scale), fnat, c.links);
    });
    return cudaGetLastError();
}

cudaError_t launch_moments(const LaunchCtx& c, int layout, const void* f, void* rho, void* u, int out_f64) {
    return dispatch(c, [&]<int Q, class S, bool W>() { return moments_impl<Q, S, W>(c, layout, f, rho, u, out_f64); });
}

cudaError_t launch_write_state(const LaunchCtx& c, int layout, const double* fnat, int uniform, void* f) {
    return dispatch(c, [&]<int Q, class S, bool W>() { return write_impl<Q, S, W>(c, layout, fnat, uniform, f); });
}

cudaError_t launch_read_state(const LaunchCtx& c, int layout, const void* f, double* fnat) {
    return dispatch(c, [&]<int Q, class S, bool W>() { return read_impl<Q, S, W>(c, layout, f, fnat); });
}

cudaError_t launch_rest_solid(const LaunchCtx& c, void* f) {
    return dispatch(c, [&]<int Q, class S, bool W>() {
        const dim3 blk = row_block(c.nx, c.ny);
        const dim3 grd((c.nx + blk.x - 1) / blk.x, (c.ny + blk.y - 1) / blk.y, c.nz);
        k_rest_solid<Q, S><<<grd, blk, 0, c.stream>>>(static_cast<typename S::T*>(f), geom(c), c.links);
        return cudaGetLastError();
    });
}

// ---------------------------------------------------------------------------
// small utilities
// ---------------------------------------------------------------------------
__global__ void k_check_unit(const float* __restrict__ v, size_t n, int* bad) {
    int local = 0;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        const float a = v[i];
        if (!(a >= 0.0f && a <= 1.0f)) ++local;  // NaN fails both comparisons
    }
    if (local) atomicAdd(bad, local);
}

__global__ void k_fill_f32(float* v, size_t n, float value) {
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
        v[i] = value;
}

static unsigned grid_1d(size_t n) {
    size_t b = (n + 255) / 256;
    if (b > 152 * 16) b = 152 * 16;
    if (b == 0) b = 1;
    return (unsigned)b;
}

cudaError_t launch_check_unit_interval(const float* v, size_t n, int* bad, cudaStream_t s) {
    k_check_unit<<<grid_1d(n), 256, 0, s>>>(v, n, bad);
    return cudaGetLastError();
}

cudaError_t launch_fill_f32(float* v, size_t n, float value, cudaStream_t s) {
    k_fill_f32<<<grid_1d(n), 256, 0, s>>>(v, n, value);
    return cudaGetLastError();
}

cudaError_t launch_fill_bytes0(void* p, size_t bytes, cudaStream_t s) { return cudaMemsetAsync(p, 0, bytes, s); }

size_t storage_bytes(int storage) {
    switch (storage) {
        case 0: return 8;
        case 1: return 4;
        case 2: return 2;
        case 3: return 2;
    }
    return 0;
}

}  // namespace hlbm
