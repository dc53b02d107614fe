// FP64 diagnostics of a state (mass, momentum, plane flux, apparent permeability,
// residual, largest velocity).
#include "dispatch.cuh"
#include "diag.cuh"

namespace hlbm {

// Block of the reductions: their partition (and so the order of their sums) is part of the result.
static dim3 block_for(int nx) {
    int bx = ((nx + 31) / 32) * 32;
    if (bx > 128) bx = 128;
    return dim3(bx, 256 / bx, 1);
}

// ---------------------------------------------------------------------------
// FP64 diagnostics. Stage 1: each block folds its cells (256 threads over x
// rows, kReduceZ z planes per thread) into 8 doubles (sum drho, sum rho*u
// (3), plane flux, 0, max|du|, max|u|) in a fixed order (diag.cuh). Stage 2:
// one block per column folds the block rows in a fixed order. The result does
// not depend on scheduling.
//
// The first version (64-bit indices, the layout chosen per direction at run
// time, residual reference loads ordered behind the previous component's
// store, one cell per thread) was latency-bound at 0.87 TB/s; 32-bit indices
// with the two-lattice layout fixed at compile time and all loads issued
// before any store bring the cell work to the copy bandwidth.
// ---------------------------------------------------------------------------
constexpr int kReduceZ = 4;

// LAY: the state's layout with 32-bit indices, or -1 (any layout, 64-bit indices).
// Measured, in-place BF16 192^3, with the final fold: 270 us with the layout chosen
// at run time, 158 us with it in the template. Also tried: a thread per cell with the four planes
// added through shared memory (64^3 13.3 vs 9.0 us, 256^3 594 vs 294: fewer resident
// warps), and the final fold in the last block to finish instead of a second launch
// (64^3 11.0 vs 10.3 us, 256^3 330 vs 312: a fence and a ticket per block).
template <int Q, class S, bool WALLS, int LAY>
__global__ void __launch_bounds__(256)
k_reduce_partials(const typename S::T* __restrict__ f, int lay, Geometry g, Phys<typename S::C> ph,
                  typename S::C inv_s, typename S::C* __restrict__ u_prev, int update_prev,
                  double* __restrict__ partials, const float* __restrict__ varpi, int drag,
                  const unsigned* __restrict__ links) {
    using C = typename S::C;
    using I = typename std::conditional<LAY >= 0, int, long long>::type;
    __shared__ DiagShared sh;
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y * blockDim.y + threadIdx.y;
    DiagCell<C> a;
    a.shifted = drag != 0;
    if (x < g.nx && y < g.ny) {
        const I N = (I)g.N;
        const int z0 = blockIdx.z * kReduceZ;
        const int z1 = z0 + kReduceZ < g.nz ? z0 + kReduceZ : g.nz;
        for (int z = z0; z < z1; ++z) {
            const I cell = (I)x + (I)g.nx * ((I)y + (I)g.ny * (I)z);
            const unsigned lm = links ? links[cell] : 0u;
            if (lm & kSolidBit) {
                // resolved obstacle: rho = 1, u = 0 (contributes nothing but its residual reference)
                if (update_prev)
                    for (int k = 0; k < 3; ++k) u_prev[(I)k * N + cell] = C(0);
                continue;
            }
            const Nbr<I> nb(g, x, y, z, lm);
            C d[Q];
#pragma unroll
            for (int i = 0; i < Q; ++i)
                d[i] = S::load(f, gather_index<Q, WALLS>(g, nb, cell, i, LAY >= 0 ? LAY : lay), inv_s);
            C up[3];
#pragma unroll
            for (int k = 0; k < 3; ++k) up[k] = u_prev[(I)k * N + cell];
            C drho, jx, jy, jz;
            moments<Q, C>(d, drho, jx, jy, jz);
            C u3[3];
            const C vp = drag ? C(varpi[cell]) : C(1);
            velocity_form<C>(jx, jy, jz, C(1) + drho, vp, drag, ph, u3[0], u3[1], u3[2]);
            a.fluid += 1;
            a.p[0] += drho;
            C mx = jx, my = jy, mz = jz;
            if (drag) {  // rho*u = (j + F/2) / (1 + lam/2)
                const C hd = C(1) / fma_(C(0.5), (C(1) - vp) * ph.omega, C(1));
                mx = fma_(C(0.5), ph.Fx, jx) * hd;
                my = fma_(C(0.5), ph.Fy, jy) * hd;
                mz = fma_(C(0.5), ph.Fz, jz) * hd;
            }  // else rho*u = j + F/2, the F/2 added per block from the fluid-cell count
            a.p[1] += mx;
            a.p[2] += my;
            a.p[3] += mz;
            if (x == g.nx - 1) {
                a.plane += 1;
                a.p[4] += mx;
            }
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                a.du = nan_max(a.du, C(fabs(u3[k] - up[k])));
                a.um = nan_max(a.um, C(fabs(u3[k])));
            }
            if (update_prev)
#pragma unroll
                for (int k = 0; k < 3; ++k) u_prev[(I)k * N + cell] = u3[k];
        }
    }
    const size_t b = blockIdx.x + (size_t)gridDim.x * (blockIdx.y + (size_t)gridDim.y * blockIdx.z);
    diag_fold<C>(a, sh, threadIdx.x + blockDim.x * threadIdx.y, blockDim.x * blockDim.y, (double)ph.Fx,
                 (double)ph.Fy, (double)ph.Fz, partials + b * 8);
}

// Block k folds column k of the partials; block 1 also forms k_app.
__global__ void __launch_bounds__(256)
k_reduce_final(const double* partials, size_t nblocks, double cells, double nu, double Fx, double* out8) {
    __shared__ double buf[256];
    const int k = blockIdx.x;
    if (k == 5) {
        return;  // column 5 is k_app, written by block 1
    }
    const double v = fold_column(partials, nblocks, k, buf);
    if (threadIdx.x == 0) {
        if (k == 0) {
            out8[0] = cells + v;  // mass = sum (1 + drho)
        } else {
            out8[k] = v;
            if (k == 1) out8[5] = (Fx != 0.0) ? nu * (v / cells) / Fx : 0.0;
        }
    }
}

size_t reduce_partials_count(const LaunchCtx& c) {
    const dim3 blk = block_for(c.nx);
    return (size_t)((c.nx + blk.x - 1) / blk.x) * ((c.ny + blk.y - 1) / blk.y) * ((c.nz + kReduceZ - 1) / kReduceZ);
}

bool reduce_grid_fits(const LaunchCtx& c) {
    const dim3 blk = block_for(c.nx);
    return (size_t)(c.ny + blk.y - 1) / blk.y <= 65535 && (size_t)(c.nz + kReduceZ - 1) / kReduceZ <= 65535 &&
           (size_t)(c.nx + blk.x - 1) / blk.x <= 0x7fffffff;
}

template <int Q, class S, bool WALLS>
static cudaError_t reduce_impl(const LaunchCtx& c, int lay, const void* f, void* u_prev, int upd,
                               double* partials, double* out8) {
    using C = typename S::C;
    const Geometry g = geom(c);
    const dim3 blk = block_for(c.nx);
    const dim3 grd((c.nx + blk.x - 1) / blk.x, (c.ny + blk.y - 1) / blk.y, (c.nz + kReduceZ - 1) / kReduceZ);
    const auto* fs = static_cast<const typename S::T*>(f);
    C* up = static_cast<C*>(u_prev);
    with_layout((size_t)Q * g.N, lay, [&]<int LAY>() {
        k_reduce_partials<Q, S, WALLS, LAY><<<grd, blk, 0, c.stream>>>(fs, lay, g, phys<C, Q>(c), C(1.0 / c.scale), up, upd,
                                                                       partials, c.varpi, c.drag, c.links);
    });
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_reduce_final<<<8, 256, 0, c.stream>>>(partials, reduce_partials_count(c), (double)g.N,
                                            (c.tau - 0.5) / 3.0, c.F[0], out8);
    return cudaGetLastError();
}

cudaError_t launch_reduce(const LaunchCtx& c, int layout, const void* f, void* u_prev, int update_prev,
                          double* partials, double* out8) {
    return dispatch(c, [&]<int Q, class S, bool W>() {
        return reduce_impl<Q, S, W>(c, layout, f, u_prev, update_prev, partials, out8);
    });
}

}  // namespace hlbm
