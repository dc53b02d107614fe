// Two D3Q19 time steps in one pass over memory (FP32, two-lattice pull streaming,
// periodic lattices whose state is larger than L2).
//
// A single step is bound by HBM: it reads and writes the whole state. This kernel
// reads the state of step n and writes the state of step n + 2; the state of
// step n + 1 lives in shared memory only. A block owns an output tile of 32 x 7 or
// 24 x 9 cells in (x, y) and marches along z. For every plane p it
//  1. copies the rows that plane p pulls from into a staging buffer (16-byte
//     asynchronous copies, one plane ahead), pulls and collides the n + 1 populations
//     of the tile and a halo of one cell (phase 1), and
//  2. pulls the populations of plane p - 1 from the n + 1 planes in shared memory,
//     collides and stores them (phase 2).
// Populations that travel up (c_z = +1) are needed two planes later, those with
// c_z = 0 one plane later and those with c_z = -1 at once, so shared memory holds
// 3, 2 and 1 planes of them: 5*3 + 9*2 + 5*1 = 38 values per cell, and 21 staged.
//
// A thread owns two neighbouring cells (lane type F2) in both phases. Phase 1 uses
// the pairs (x0 - 1, x0), (x0 + 1, x0 + 2), ...: with x0 even the x-shifted
// directions are aligned pairs in the staged rows; phase 2 uses (x0, x0 + 1), ...,
// whose x-shifted directions are aligned pairs in the n + 1 planes. The
// directions with c_x = 0 would then be read at stride two: their n + 1 planes keep
// even and odd columns apart, so both accesses are free of bank conflicts.
//
// The collision is the function of the single-step kernels, so two steps here and
// two single steps give the same bits.
//
// What bounds it: no longer HBM alone. Two steps of 256^3 move 2.68 GB (0.40 ms at the copy
// rate) and take 0.62 ms: shared memory allows 15 warps per SM, whose copies, collisions and
// shared-memory accesses add up more than they overlap (DRAM 51 %, shared memory 41 % busy), and
// phase 1 works on 1.32 to 1.37 times the cells. With parts switched off at 192^3 (us per step,
// complete 136): no copies 103, no stores 115, collisions passed through 124, none of the three
// 49. Measured against the single-step kernel, us per step: 256^3 373 -> 309, 192^3 160 -> 137,
// 288^3 533 -> 420, 240^3 309 -> 250, 128^3 49.5 -> 44.2, 160^3 94.8 -> 83.6; single steps run at
// 1.02 of the copy rate.
// Variants that were slower at 256^3: two larger blocks per SM with the whole
// window in registers 340, one tensor-map box per direction 341, a bulk copy per row 386,
// delay lines in registers 337, and every 16-bit variant (bound by instructions).
#include "k_step_pair.cuh"
#include "step2_plan.h"

namespace hlbm {

namespace {

using L = Lat<19>;

constexpr int kBlocksPerSM = kStep2BlocksPerSM;

// Position of direction i within the directions of the same c_z, in index order, and
// the first position of a c_z group in the staging buffer (up, flat, down).
__host__ __device__ constexpr int group_pos(int i) {
    int n = 0;
    for (int j = 0; j < i; ++j) n += L::cz(j) == L::cz(i);
    return n;
}
__host__ __device__ constexpr int group_first(int cz) { return cz > 0 ? 0 : (cz == 0 ? 5 : 14); }
struct StagedDirs {
    signed char dir[19], cy[19];
    constexpr StagedDirs() : dir(), cy() {
        for (int i = 0; i < 19; ++i) {
            const int k = group_first(L::cz(i)) + group_pos(i);
            dir[k] = (signed char)i;
            cy[k] = (signed char)L::cy(i);
        }
    }
};
__constant__ const StagedDirs kStaged;

// Output tile of TX x TY columns.
template <int TX, int TY>
struct Tile {
    static constexpr int EX = TX + 2, EY = TY + 2;  // with its halo
    static constexpr int PX = EX / 2;               // pairs per extended row
    static constexpr int kPairs = PX * EY;
    static constexpr int kThreads = (kPairs + 31) / 32 * 32;
    static constexpr int PS = EX * EY;  // values of one direction of one n + 1 plane
    static constexpr int C = 4;         // floats per 16-byte chunk
    static constexpr int kChunks = TX / C + 2, SX = kChunks * C;  // staged columns x0 - C .. x0 + TX + C - 1
    static constexpr int kStage = 19 * SX * EY, kUp = 15 * PS, kFlat = 18 * PS, kDown = 5 * PS;  // floats
    static constexpr int kBytes = (kStage + kUp + kFlat + kDown) * (int)sizeof(float);
    static_assert(TX % C == 0 && kChunks <= 32 && kBlocksPerSM * (kBytes + 1024) <= 228 * 1024, "tile");
};

struct Pops {
    F2 v[19];
    __device__ __forceinline__ F2 operator[](int i) const { return v[i]; }
};
__device__ __forceinline__ F2 ld2(const float* a) {
    const float2 f = *reinterpret_cast<const float2*>(a);
    return F2(f.x, f.y);
}

// Porosity of a pair of cells (scalar, or the diagonal tensor).
template <int FORM>
struct Porosity {
    static constexpr int kN = FORM == FORM_ANISO ? 3 : 1;
    F2 v[kN];
    __device__ __forceinline__ void load(const float* varpi, int N, int a, int b) {
#pragma unroll
        for (int k = 0; k < kN; ++k) v[k] = F2(__ldg(varpi + k * N + a), __ldg(varpi + k * N + b));
    }
};
template <int FORM, class Sink>
__device__ __forceinline__ void collide_pair(const Pops& d, const Porosity<FORM>& w, const Phys<float>& ph, Sink out) {
    if constexpr (FORM == FORM_ANISO) collide_aniso<19, F2, false>(d, w.v[0], w.v[1], w.v[2], ph, 1.0f, 1.0f, out);
    else if constexpr (FORM == FORM_DRAG) collide_drag<19, F2, false>(d, w.v[0], ph, 1.0f, 1.0f, out);
    else collide<19, F2, false, FORM == FORM_SHIFT_FX>(d, w.v[0], ph, 1.0f, 1.0f, out);
}

__device__ __forceinline__ void copy16(unsigned dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ int wrap1(int v, int n) { return v < 0 ? v + n : (v >= n ? v - n : v); }

// zc: output planes per block. varpi: [cells], or [3][cells] for the tensor form.
template <int FORM, int TX, int TY>
__global__ void __launch_bounds__(Tile<TX, TY>::kThreads, kBlocksPerSM)
k_step2(const float* __restrict__ fin, float* __restrict__ fout, const float* __restrict__ varpi, Geometry g,
        Phys<float> ph, int zc) {
    using K = Tile<TX, TY>;
    constexpr int EX = K::EX, EY = K::EY, PX = K::PX, PS = K::PS, C = K::C, SX = K::SX;
    constexpr int kThreads = K::kThreads, kChunks = K::kChunks;
    extern __shared__ __align__(16) float smem[];
    float* const up = smem + K::kStage;
    float* const flat = up + K::kUp;
    float* const down = flat + K::kFlat;
    const int N = (int)g.N, plane = g.nx * g.ny;
    const int t = threadIdx.x;
    const int x0 = blockIdx.x * TX, y0 = blockIdx.y * TY, z0 = blockIdx.z * zc;
    const int xe = min(x0 + TX, g.nx), ye = min(y0 + TY, g.ny), z1 = min(z0 + zc, g.nz);

    // phase 1: the pair at extended position (2 px, py), cells x0 - 1 + 2 px and the next
    const int py = t / PX, px = t - py * PX;
    const int ya = y0 - 1 + py;
    const bool on1 = t < K::kPairs && x0 - 1 + 2 * px <= xe && ya <= ye;
    const int row1 = wrap1(ya, g.ny) * g.nx;
    const int a1 = row1 + wrap1(x0 - 1 + 2 * px, g.nx), b1 = row1 + wrap1(x0 + 2 * px, g.nx);
    const int w1 = py * EX + 2 * px;  // where the pair lands in an n + 1 plane
    // phase 2: the pair at output position (2 qx, qy)
    const int qy = t / (TX / 2), qx = t - qy * (TX / 2);
    const int xo = x0 + 2 * qx, yo = y0 + qy;
    const bool on2 = qy < TY && xo < xe && yo < ye;
    const int cell2 = yo * g.nx + xo;
    const int w2 = (qy + 1) * EX + 2 * qx + 1;

    // The staged rows of the directions with the same c_z come from one z plane; a row is kChunks
    // 16-byte chunks, a warp copies kRows rows at once, and a thread keeps the offsets of its chunks
    // within that plane's set of directions (-1: nothing to copy).
    constexpr int kRows = 32 / kChunks, kStride = kRows * (kThreads / 32);
    constexpr int nU = (5 * EY + kStride - 1) / kStride, nF = (9 * EY + kStride - 1) / kStride;
    const int lane = t & 31, lr = lane / kChunks, lc = lane - lr * kChunks;
    const int xs = wrap1(x0 + (lc - 1) * C, g.nx);
    const bool copies = lr < kRows && x0 + (lc - 1) * C <= xe + 1;  // up to the last column that is pulled from
    const int srow = (t >> 5) * kRows + lr;
    const unsigned stage = (unsigned)__cvta_generic_to_shared(smem) + (srow * SX + lc * C) * 4;
    int off[2 * nU + nF];
    const auto offset_of = [&](int first, int count, int r) {
        const int k = r / EY, y = r - k * EY;
        if (!copies || k >= count || y >= ye - y0 + 2) return -1;
        return kStaged.dir[first + k] * N + wrap1(y0 - 1 + y - kStaged.cy[first + k], g.ny) * g.nx + xs;
    };
#pragma unroll
    for (int k = 0; k < nU; ++k) {
        off[k] = offset_of(0, 5, srow + k * kStride);
        off[nU + nF + k] = offset_of(14, 5, srow + k * kStride);
    }
#pragma unroll
    for (int k = 0; k < nF; ++k) off[nU + k] = offset_of(5, 9, srow + k * kStride);
    const auto fetch = [&](int p) {
        const int z = wrap1(p, g.nz);
#pragma unroll
        for (int k = 0; k < 2 * nU + nF; ++k) {
            const int cz = k < nU ? 1 : (k < nU + nF ? 0 : -1), kk = cz > 0 ? k : (cz == 0 ? k - nU : k - nU - nF);
            const float* const base = fin + wrap1(z - cz, g.nz) * plane;
            if (off[k] >= 0) copy16(stage + (group_first(cz) * EY + kk * kStride) * (SX * 4), base + (unsigned)off[k]);
        }
    };

    Porosity<FORM> v1;  // of the phase 1 pair, loaded a plane ahead
    fetch(z0 - 1);
    if (on1) v1.load(varpi + wrap1(z0 - 1, g.nz) * plane, N, a1, b1);
    int pu = 0;  // up[] buffer of the plane being written: cycles through 3
#pragma unroll 1
    for (int p = z0 - 1; p <= z1; ++p) {
        const int pf = (p - z0 + 1) & 1;  // flat[] buffer of plane p
        Porosity<FORM> v2;
        if (p > z0 && on2) v2.load(varpi + (p - 1) * plane, N, cell2, cell2 + 1);
        // the staged rows have landed, and phase 2 of the previous plane has read its slots
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncthreads();
        if (on1) {
            const float* const w = smem + py * SX + 2 * px + C - 1;
            Pops d;
#pragma unroll
            for (int i = 0; i < 19; ++i) {
                const float* const a = w + (group_first(L::cz(i)) + group_pos(i)) * (EY * SX);
                d.v[i] = L::cx(i) == 0 ? F2(a[0], a[1]) : ld2(L::cx(i) > 0 ? a - 1 : a + 1);
            }
            float* const uw = up + pu * (5 * PS) + w1;
            float* const fw = flat + pf * (9 * PS) + w1;
            float* const dw = down + w1;
            collide_pair<FORM>(d, v1, ph, [&](int i, F2 v) {
                float* const a = (L::cz(i) > 0 ? uw : (L::cz(i) == 0 ? fw : dw)) + group_pos(i) * PS;
                const float2 f = v.split();
                if (L::cx(i) == 0) {  // even columns, then odd columns
                    a[-px] = f.x;
                    a[-px + PX] = f.y;
                } else {
                    *reinterpret_cast<float2*>(a) = f;
                }
            });
        }
        __syncthreads();
        if (p < z1) {
            fetch(p + 1);
            if (on1) v1.load(varpi + wrap1(p + 1, g.nz) * plane, N, a1, b1);
        }
        const int pu1 = pu == 0 ? 2 : pu - 1, pu2 = pu1 == 0 ? 2 : pu1 - 1;  // up[] of the planes p - 1 and p - 2
        if (p > z0 && on2) {
            const float* const ur = up + pu2 * (5 * PS) + w2;
            const float* const fr = flat + (pf ^ 1) * (9 * PS) + w2;
            const float* const dr = down + w2;
            Pops e;
#pragma unroll
            for (int i = 0; i < 19; ++i) {
                const float* const a = (L::cz(i) > 0 ? ur : (L::cz(i) == 0 ? fr : dr)) + (group_pos(i) * PS - L::cy(i) * EX);
                e.v[i] = L::cx(i) == 0 ? F2(a[PX - 1 - qx], a[-qx]) : ld2(L::cx(i) > 0 ? a - 1 : a + 1);
            }
            float* const o = fout + ((p - 1) * plane + cell2);
            collide_pair<FORM>(e, v2, ph, [&](int i, F2 v) { *reinterpret_cast<float2*>(o + i * N) = v.split(); });
        }
        pu = pu == 2 ? 0 : pu + 1;
    }
}

template <int FORM, int TX, int TY>
cudaError_t step2_tile(const LaunchCtx& c, int zc, const void* fin, void* fout, const float* varpi) {
    using K = Tile<TX, TY>;
    const auto kern = k_step2<FORM, TX, TY>;
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, K::kBytes);
    if (e != cudaSuccess) return e;
    const Geometry g{c.nx, c.ny, c.nz, 0, 0, 0, (size_t)c.nx * c.ny * c.nz};
    const dim3 grd((c.nx + TX - 1) / TX, (c.ny + TY - 1) / TY, (c.nz + zc - 1) / zc);
    kern<<<grd, K::kThreads, K::kBytes, c.stream>>>(static_cast<const float*>(fin), static_cast<float*>(fout),
                                                    FORM == FORM_ANISO ? c.varpi3 : varpi, g,
                                                    make_phys<float, 19>(c.tau, c.F), zc);
    return cudaGetLastError();
}
template <int FORM>
cudaError_t step2_impl(const LaunchCtx& c, const void* fin, void* fout, const float* varpi) {
    const Step2Plan p = step2_plan(c);
    return p.wide ? step2_tile<FORM, 32, 7>(c, p.zc, fin, fout, varpi) : step2_tile<FORM, 24, 9>(c, p.zc, fin, fout, varpi);
}

}  // namespace

// Periodic FP32 lattices whose rows are whole 16-byte chunks, with 32-bit indices and axes
// that one wrap correction covers, and whose two states are well above L2 (228 MB: at
// 96^3 one step per pass is faster, 21.0 vs 23.0 us). The gain follows step2_plan's `useful`;
// over 60 lattices of 1.2 to 25 M cells it was 1.05 to 1.30 above these limits for a force along
// x, 1.02 to 1.25 for other forces and drag, 1.03 to 1.17 for the tensor, which loads three
// porosities; below them 0.97 to 1.11, 0.98 to 1.10 and 0.92 to 1.04.
bool step2_applies(const LaunchCtx& c) {
    const size_t n = (size_t)c.nx * c.ny * c.nz;
    if (c.variant != 0 || c.q != 19 || c.storage != 1 || c.wall[0] || c.wall[1] || c.wall[2] || c.links || c.nx % 4 != 0 ||
        c.nx < 8 || c.ny < 4 || c.nz < 4 || 19 * n >= ((size_t)1 << 31) || n < 1500000)
        return false;
    const int form = step_form(c, 19);
    const double need = form == FORM_SHIFT_FX ? 0.78 : (form == FORM_ANISO ? 0.86 : 0.83);
    return step2_plan(c, need).useful >= need;
}

cudaError_t launch_step2(const LaunchCtx& c, const void* fin, void* fout, const float* varpi) {
    switch (step_form(c, 19)) {
        case FORM_SHIFT_FX: return step2_impl<FORM_SHIFT_FX>(c, fin, fout, varpi);
        case FORM_SHIFT: return step2_impl<FORM_SHIFT>(c, fin, fout, varpi);
        case FORM_DRAG: return step2_impl<FORM_DRAG>(c, fin, fout, varpi);
        default: return step2_impl<FORM_ANISO>(c, fin, fout, varpi);
    }
}

}  // namespace hlbm
