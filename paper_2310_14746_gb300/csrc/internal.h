// Internal interface between the C ABI (api.cu) and the kernel translation
// units. Not installed; callers use include/hlbm.h.
#pragma once

#include <cuda_runtime.h>
#include <atomic>
#include <cstddef>
#include <cstdint>
#include <utility>

namespace hlbm {

enum Chain { CHAIN_NONE = 0, CHAIN_GRAPH = 1, CHAIN_STREAM = 2 };  // captured into a graph / launched one by one
enum StepMode { MODE_TWO_LATTICE = 0, MODE_AA_EVEN = 1, MODE_AA_ODD = 2 };

// Everything a launch needs to know about a lattice, in plain types.
struct LaunchCtx {
    int q;          // 9 or 19
    int storage;    // HLBM_F64 / F32 / F16DEV / BF16DEV
    int nx, ny, nz;
    int wall[3];    // 1 = half-way bounce-back on that axis
    double tau;
    double F[3];
    double scale;   // storage scale s (deviations are stored times s)
    cudaStream_t stream;
    int drag = 0;                  // homogenization form: 0 equilibrium shift, 1 explicit drag
    const float* varpi = nullptr;  // porosity control (observables need it in the drag form)
    const float* varpi3 = nullptr; // diagonal porosity tensor [3][cells], or null (isotropic)
    const unsigned* links = nullptr; // solid-link masks (resolved obstacles), or null
    int variant = 0;                 // 0: fastest applicable step kernel; 1: per-cell kernel only
    int chained = CHAIN_NONE;        // is the kernel before one of the same run? (see launch_chained)
};

#ifdef __CUDACC__
// Launch of a kernel that begins with chain_wait. Where `chained`, its blocks are placed while the
// kernel before it on the stream still runs, so that its launch costs no time between the two.
// Only for a kernel that directly follows another kernel on its stream, or in its graph: the first
// kernel of a graph, or one that follows a graph or a copy, is launched plainly (with the attribute
// such kernels have been seen to start before that work had ended). So chained kernels only go to
// streams and graphs that the library alone launches into.
// Measured, us per step in a graph of 16, plain -> chained: FP32 24^3 2.05 -> 1.69, 32^3 2.43 ->
// 2.05, 64^3 5.51 -> 5.23, 96^3 20.8 -> 20.3; FP16 32^3 2.56 -> 2.05, 48^3 3.20 -> 2.69. Where two
// grids do not fit the chip together, but one leaves room, the early blocks crowd the SMs that are
// free first, and the others stay idle: 45^3 (0.68 of the blocks that fit) 3.64 -> 3.99, 41x44x39
// with walls (0.56) 4.23 -> 5.10, but 36^3 (0.43) 3.07 -> 2.69 and 51^3 (0.87) 4.72 -> 4.36. So grids
// between 0.44 and 0.78 are launched plainly in a graph (one by one, where the gaps are
// longer, chained: 48^3 gradient 1.60 against 1.87 ms).
// Launched one by one, a 48^3 gradient over 90 steps takes 1.60 instead of 2.10 ms.
template <class... P, class... A>
cudaError_t launch_chained(int chained, void (*kern)(P...), dim3 grd, dim3 blk, size_t smem, cudaStream_t s, A&&... args) {
    if (chained == CHAIN_GRAPH) {
        int fit = 0;  // blocks per SM
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&fit, kern, (int)(blk.x * blk.y * blk.z), smem) == cudaSuccess) {
            const double share = (double)grd.x * grd.y * grd.z / (152.0 * fit);
            if (share > 0.44 && share < 0.78) chained = CHAIN_NONE;
        }
    }
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grd;
    cfg.blockDim = blk;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = chained ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kern, P(std::forward<A>(args))...);
}
// Waits until the kernel before has ended and its stores are visible, then lets the next kernel's
// blocks be placed: at most two kernels overlap, and every load of the caller happens after the
// end of the kernel that wrote its operands. `x` takes part in every address, so no load can be
// moved before the wait.
__device__ __forceinline__ void chain_wait(int& x) {
    asm volatile("griddepcontrol.wait;\n\tgriddepcontrol.launch_dependents;" : "+r"(x) : : "memory");
}
#endif

// Block of a one-thread-per-cell kernel: a whole row of x as long as it fits 256
// threads (at least 128 threads), a longer row in equal pieces where that leaves
// fewer idle lanes than blocks of 128 cells times two rows, the only shape before:
// those left up to 40 % of the lanes of a ragged row idle. Measured on the step,
// 128-cell blocks vs this rule, us: FP32 150x101x67 with walls 32.1 -> 28.8, 160^3
// with walls 113 -> 102, 221x143x203 163 -> 159, 256^3 376.6 -> 373.4, 128^3 49.4 ->
// 49.5, 64^3 5.81 -> 5.46, 48^3 4.10 -> 3.84, 33x41x44 4.04 -> 3.33; FP16 152x104x96
// with walls 41.2 -> 35.9. Equal pieces with as many idle lanes measured 4 % slower
// (D2Q9 329x245), so a tie keeps the old shape. So does a y axis that the rows of this rule
// would not cover with one grid: a server's lattice may have up to 131070 rows of more than 64
// cells, 262140 of up to 64 and 524280 of up to 32.
constexpr int kMaxGridY = 65535, kMaxGridZ = 65535;
inline dim3 row_block_old(int nx) {
    const int bx = nx > 96 ? 128 : (nx + 31) / 32 * 32;
    return dim3(bx, 256 / bx, 1);
}
inline long long rows_per_grid(int nx) { return (long long)kMaxGridY * row_block_old(nx).y; }
inline dim3 row_block(int nx, int ny) {
    const int pieces = (nx + 255) / 256, bx = ((nx + pieces - 1) / pieces + 31) / 32 * 32;
    const dim3 old = row_block_old(nx), blk(bx, bx >= 128 ? 1 : 128 / bx, 1);
    if (pieces > 1 && pieces * bx >= (nx + 127) / 128 * 128) return old;
    return (ny + (int)blk.y - 1) / (int)blk.y > kMaxGridY ? old : blk;
}

// Block of a paired kernel (x in cell pairs): about 128 threads that leave the fewest
// idle lanes over the lattice, counting the row tail, the partly filled warp of a
// block and the tail of y. Candidate widths: 64, 32 and 16 pairs, and the row cut into
// one to four equal pieces (any width: a warp may span rows). Before, blocks had 256
// threads and widths of 32, 64, 96 or 128 pairs. Measured, us per step before -> with
// this rule: two-lattice FP16 96^3 15.4 -> 12.0, 160^3 63.1 -> 55.8, 42x50x60 4.35 ->
// 3.59, 64^3 5.12 -> 4.61, 192^3 94.5 -> 92.8, 256^3 216.3 -> 214.1, 384x192x192 184.4 ->
// 182.0; BF16 160^3 57.3 -> 53.2, 176x176x152 (drag) 70.9 -> 67.8, 204x190x180 (tensor)
// 131 -> 126; in place FP16 80x64x72 8.7 -> 6.2, 160^3 63.7 -> 57.6, BF16 192^3 95.5 ->
// 93.8. Pieces of 16 pairs where nx is no multiple of 32 measured 110 instead of 91.8
// (BF16 222x144x200), hence the penalty. Where y is longer than a grid, only blocks of
// enough rows count (16 pairs times 8 rows always fit up to 524280 rows).
inline dim3 pair_block(int nx, int ny, int cap) {
    const int pairs = nx / 2, most = cap < 192 ? cap : 192;
    const int widths[] = {64, 32, 16, pairs, (pairs + 1) / 2, (pairs + 2) / 3, (pairs + 3) / 4};
    dim3 best(32, 4, 1);
    double score_best = -1.0;
    for (int bx : widths) {
        if (bx < 1 || bx > most) continue;
        for (int by = 1; bx * by <= most; ++by) {
            if ((ny + by - 1) / by > kMaxGridY) continue;
            const int threads = bx * by, lanes = (threads + 31) / 32 * 32;
            double score = (double)pairs / ((pairs + bx - 1) / bx) * by / lanes * ny / ((ny + by - 1) / by * by);
            if (threads < 64) score *= 0.8;            // too few warps per block to fill an SM
            if (bx < 32 && bx < pairs) score *= nx % 32 == 0 ? 0.97 : 0.85;  // short pieces, worse when they straddle lines
            score -= 1e-4 * (threads < 128 ? 128 - threads : threads - 128) / 128;
            if (score > score_best) {
                score_best = score;
                best = dim3(bx, by, 1);
            }
        }
    }
    return best;
}

// Solid-link masks from a solid flag per cell (uint8, nonzero = solid): bit i of
// links[cell] is set when the pull source x - c_i is solid (periodic wrap; a
// source beyond a domain wall is left to the wall logic), bit 31 when the
// cell itself is solid.
cudaError_t launch_build_links(const LaunchCtx& c, const unsigned char* solid, unsigned* links);

// One time step: read `fin` in the layout implied by `mode`, write `fout`
// (== fin for the AA modes).
cudaError_t launch_step(const LaunchCtx& c, int mode, const void* fin, void* fout,
                        const float* varpi);
// Two steps of a two-lattice state in one launch (k_step2.cu), where step2_applies.
bool step2_applies(const LaunchCtx& c);
cudaError_t launch_step2(const LaunchCtx& c, const void* fin, void* fout, const float* varpi);

// Many time steps of a small two-lattice state in one launch, in place on `f`
// (NATURAL layout), with the state resident in the shared memory of one
// thread-block cluster: the same bits as nsteps MODE_TWO_LATTICE steps.
// resident_applies says whether the lattice fits (on the current device).
bool resident_applies(const LaunchCtx& c);
cudaError_t launch_resident(const LaunchCtx& c, void* f, const float* varpi, int nsteps);

// Moments of a state stored in `layout` (Layout enum of lattice.cuh). rho
// and/or u may be null. out_f64 selects double outputs, else float.
cudaError_t launch_moments(const LaunchCtx& c, int layout, const void* f, void* rho, void* u,
                           int out_f64);

// Per-block FP64 partials of the diagnostics, then a fixed-order final
// reduction (one block per quantity) into out8[8] (device). u_prev (arithmetic type of the
// storage: double for F64, float otherwise; 3*cells) is compared against and,
// if update_prev, overwritten. `partials` is caller-provided scratch of at
// least reduce_partials_count(c) * 8 doubles.
size_t reduce_partials_count(const LaunchCtx& c);
// Whether the partials kernel's grid for this lattice is within the launch limits.
bool reduce_grid_fits(const LaunchCtx& c);
cudaError_t launch_reduce(const LaunchCtx& c, int layout, const void* f, void* u_prev,
                          int update_prev, double* partials, double* out8);

// Write the natural post-collision populations fnat (FP64 full values) into
// the state buffer in `layout`. fnat is [q][cells] when uniform == 0, or q
// values applied to every cell when uniform == 1.
cudaError_t launch_write_state(const LaunchCtx& c, int layout, const double* fnat, int uniform,
                               void* f);
// Rest populations into the solid cells (c.links) of a state buffer in any layout.
cudaError_t launch_rest_solid(const LaunchCtx& c, void* f);
// Read the state as natural FP64 full populations [q][cells].
cudaError_t launch_read_state(const LaunchCtx& c, int layout, const void* f, double* fnat);

// Count values outside [0, 1] (or NaN) into *bad (device int, accumulated).
cudaError_t launch_check_unit_interval(const float* v, size_t n, int* bad, cudaStream_t s);
cudaError_t launch_fill_f32(float* v, size_t n, float value, cudaStream_t s);
cudaError_t launch_fill_bytes0(void* p, size_t bytes, cudaStream_t s);

size_t storage_bytes(int storage);

// A yes or no about the current context (a context may be confined to a part of its device, so a
// device's answer need not hold in it), asked when the context is not the one of the last answer.
// `ask` returns 1 or 0, or -1 when it could not tell: that counts as no and is not remembered.
struct ContextFact {
    std::atomic<unsigned long long> known[64] = {};  // per device: context id * 2 + answer
    bool get(int (*ask)());
};

// Memory kept between objects, in the current context (mem.cu). A pool belongs to one handle at
// a time; every block taken from it is freed, and its streams are drained, before it is released.
bool pool_keeps(size_t bytes);  // does a released pool keep this much mapped?
cudaError_t pool_acquire(cudaMemPool_t* pool);
void pool_release(cudaMemPool_t pool);
// The servers' pool; where nothing is kept, a new one that the caller destroys (own).
cudaError_t pool_shared(cudaMemPool_t* pool, bool* own);
// A stream for the length of a call. Released with `idle` when it has been waited for, and not
// when that failed (within a capture): it is then destroyed.
cudaError_t stream_acquire(cudaStream_t* s);
void stream_release(cudaStream_t s, bool idle);
cudaError_t pool_alloc(cudaMemPool_t pool, void** p, size_t bytes, cudaStream_t s);
cudaError_t device_malloc(void** p, size_t bytes);  // cudaMalloc, for blocks that no pool should hold
void* pinned_acquire(size_t bytes, size_t* capacity);  // null: out of memory
void pinned_release(void* b, size_t capacity);
double* slot_acquire();  // 64 bytes of pinned memory, or null
void slot_release(double* p);
void memory_give_back();  // return what is kept for later objects

// All n values in [0, 1] (NaN fails)? The input may be a whole lattice (64 MiB
// at 256^3), so the test runs in blocks without an early exit inside a block:
// the inner loop vectorises, and a bad value still stops the scan at the end
// of its block.
inline bool host_unit_interval(const float* v, size_t n) {
    constexpr size_t kBlock = 4096;
    for (size_t b = 0; b < n; b += kBlock) {
        const size_t e = b + kBlock < n ? b + kBlock : n;
        int good = 1;
        for (size_t k = b; k < e; ++k) good &= (v[k] >= 0.0f) & (v[k] <= 1.0f);
        if (!good) return false;
    }
    return true;
}

// Reverse step of the outflow-flux adjoint: fn is the forward state before the
// step (NATURAL layout), lam_in = dJ/df^{n+1} and lam_out = dJ/df^n ([q][cells]
// FP32, distinct buffers); grad (FP32 cells) accumulates dJ/dvarpi.
cudaError_t launch_adjoint_step(const LaunchCtx& c, const void* fn, const float* lam_in, float* lam_out,
                                const float* varpi, float* grad);
// dJ/df of the final state for J = sum over the plane x = plane_x of rho*u_x.
cudaError_t launch_flux_seed(const LaunchCtx& c, float* lam, int plane_x);
// J of a state in `layout` into out (one double, device).
cudaError_t launch_plane_flux(const LaunchCtx& c, int layout, const void* f, int plane_x, double* out);

}  // namespace hlbm
