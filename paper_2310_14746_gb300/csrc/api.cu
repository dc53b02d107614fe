// C ABI of the HBGK library (include/hlbm.h): handles, validation, state
// bookkeeping, CUDA-graph replay of step sequences, checkpoints.
#include <cuda_runtime.h>

#include <cmath>
#include <cstdio>
#include <cstring>
#include <new>
#include <vector>

#include "../../include/hlbm.h"
#include "internal.h"

using namespace hlbm;

namespace {

thread_local char g_last_cuda[256] = "";

int cuda_fail(cudaError_t e) {
    std::snprintf(g_last_cuda, sizeof(g_last_cuda), "%s: %s", cudaGetErrorName(e), cudaGetErrorString(e));
    return e == cudaErrorMemoryAllocation ? HLBM_ERR_OOM : HLBM_ERR_CUDA;
}

#define HLBM_CUDA(call)                               \
    do {                                              \
        cudaError_t e_ = (call);                      \
        if (e_ != cudaSuccess) return cuda_fail(e_);  \
    } while (0)

// Steps of the two step graphs. Even: a graph returns the state to its starting layout. A replay
// costs about 3 us beside its kernels (kernels chained, us per step, 8 / 16 / 32 / 64 steps: 32^3
// 2.31 / 2.05 / 2.01 / 1.95), and capturing and instantiating a graph about 15 us and 3 us per step,
// again after every change of a setting. So the long one is captured once kLongFrom steps have been
// asked for with the present settings (a change of the force and 24 steps of 24^3: both graphs 125
// us, the short one alone 91; and 100 steps: 254 to 258 either way), and the short one, for what the
// long one leaves, not before kShortFrom.
constexpr int kGraphSteps[] = {8, 16};
constexpr long long kLongFrom = 96, kShortFrom = 512;
// Runs of a small lattice that one resident launch takes: below kResidentMin the launch and its
// loads and stores (about 5 us) cost more than single steps; kResidentMax bounds one launch to
// about a millisecond or two.
constexpr long kResidentMin = 6, kResidentMax = 1000;
// Samples of hlbm_reduce_series per graph replay. Even, so that a replay returns the state to its
// starting layout. Launched one by one, the three kernels of a sample leave the GPU idle for about
// a third of a 64^3 sample (step 5.5, diagnostics 9 us). A series of 200 samples, us, launched /
// replayed / replayed with the diagnostics on a branch: 24^3 3290 / 2210 / 1970, 48^3 3700 /
// 2670 / 2170, 64^3 4360 / 3180 / 2490, 96^3 10180 / 8850 / 7360, 128^3 21270 / 19980 / 18330.
constexpr int kSeriesSamples = 8;
constexpr long kSeriesMin = 32;  // shorter series do not pay for the capture

// The lattice Layout enum values (lattice.cuh), repeated for host code.
constexpr int kNatural = 0, kStreamed = 1, kSwapped = 2;

}  // namespace

struct hlbm_lattice {
    int q = 19, nx = 0, ny = 0, nz = 0, storage = HLBM_F32, pattern = HLBM_TWO_LATTICE;
    int device = 0;
    cudaStream_t stream = nullptr;
    cudaStream_t cap_stream = nullptr;  // private stream used only to capture graphs
    cudaEvent_t fork_ev = nullptr;      // where a gradient leaves the handle's stream
    double tau = 1.0;
    double F[3] = {0.0, 0.0, 0.0};
    int bc[3] = {HLBM_PERIODIC, HLBM_PERIODIC, HLBM_PERIODIC};
    double scale = 1.0;
    int homog = HLBM_HOMOG_SHIFT;
    size_t cells = 0;
    void* buf[2] = {nullptr, nullptr};
    int cur = 0;     // two-lattice: buffer holding the state
    int aa_odd = 0;  // AA: 1 when the state is in the SWAPPED layout
    long long step = 0;
    float* varpi = nullptr;
    float* varpi3 = nullptr;  // diagonal porosity tensor (allocated on first use)
    int aniso = 0;
    unsigned* links = nullptr;  // solid-link masks (resolved obstacles), or null
    void* u_prev = nullptr;
    double* partials = nullptr;
    double* out8 = nullptr;
    double* out8_host = nullptr;
    cudaGraphExec_t gexec[2] = {};  // of kGraphSteps
    bool graph_valid[2] = {};       // captured with the present settings?
    long long graph_steps = 0;      // steps asked of hlbm_step with the present settings
    int chaining = CHAIN_NONE;      // of the steps that are launched next
    cudaGraphExec_t series_exec = nullptr;  // kSeriesSamples samples of hlbm_reduce_series
    int series_every = 0;                   // steps between its samples; 0: to be captured again
    cudaStream_t series_stream = nullptr;   // capture stream of its diagnostics
    cudaEvent_t series_ev[3] = {};
    void settings_changed() {
        graph_valid[0] = graph_valid[1] = false;
        graph_steps = 0;
        series_every = 0;
    }
    int step_variant = HLBM_STEP_AUTO;
    cudaMemPool_t pool = nullptr;  // scratch, and the lattice of a handle that pool_keeps() all of
    bool pooled = false;           // is this one?
    bool moved = false;            // the stream was replaced: earlier work may be on another one

    size_t state_bytes() const { return (size_t)q * cells * storage_bytes(storage); }
    size_t arith_bytes() const { return storage == HLBM_F64 ? 8 : 4; }
    int layout() const {
        if (pattern == HLBM_TWO_LATTICE) return kNatural;
        return aa_odd ? kSwapped : kStreamed;
    }
    void* state() const { return buf[pattern == HLBM_TWO_LATTICE ? cur : 0]; }
    LaunchCtx ctx(cudaStream_t s) const {
        LaunchCtx c;
        c.q = q;
        c.storage = storage;
        c.nx = nx;
        c.ny = ny;
        c.nz = nz;
        for (int a = 0; a < 3; ++a) c.wall[a] = bc[a] == HLBM_HALFWAY_BOUNCE_BACK;
        c.tau = tau;
        for (int a = 0; a < 3; ++a) c.F[a] = F[a];
        c.scale = scale;
        c.stream = s;
        c.drag = homog == HLBM_HOMOG_DRAG;
        c.varpi = varpi;
        c.varpi3 = aniso ? varpi3 : nullptr;
        c.links = links;
        c.variant = step_variant;
        c.chained = chaining;
        return c;
    }
};

namespace {

// Make the handle's device current for the duration of a call.
struct DeviceGuard {
    int prev = -1;
    explicit DeviceGuard(int dev) {
        if (cudaGetDevice(&prev) == cudaSuccess && prev != dev) cudaSetDevice(dev);
        else prev = -1;
    }
    ~DeviceGuard() {
        if (prev >= 0) cudaSetDevice(prev);
    }
};

// Temporary device memory of a call (the adjoint's checkpoints, staging buffers of host
// I/O), stream-ordered on the handle's stream, from a pool that is the handle's own while
// it lives and is kept for the next handle afterwards (mem.cu). It holds what it has
// mapped: with the default pool (release threshold 0) the 14.5 GB of checkpoints of a
// 128^3 x 2000-step gradient were unmapped at every synchronisation and mapped again by
// the next call (0.395 s vs 0.370 s per gradient).
// hlbm_release_scratch hands unused memory back.
cudaError_t scratch_alloc(hlbm_t* h, void** p, size_t bytes) {
    if (!h->pool) {
        const cudaError_t e = pool_acquire(&h->pool);
        if (e != cudaSuccess) return e;
    }
    return pool_alloc(h->pool, p, bytes, h->stream);
}

// Memory that stays for the handle's life. A small lattice takes it from the pool too:
// the next one then finds it mapped. A large one would not be kept, and maps faster without
// a pool (hlbm_create of a 384^3 FP16 lattice 2.7 ms, from a pool 5.9).
cudaError_t lattice_alloc(hlbm_t* h, void** p, size_t bytes) {
    return h->pooled ? scratch_alloc(h, p, bytes) : device_malloc(p, bytes);
}

void free_all(hlbm_t* h) {
    for (cudaGraphExec_t e : h->gexec)
        if (e) cudaGraphExecDestroy(e);
    if (h->series_exec) cudaGraphExecDestroy(h->series_exec);
    for (cudaEvent_t e : h->series_ev)
        if (e) cudaEventDestroy(e);
    if (h->series_stream) cudaStreamDestroy(h->series_stream);
    if (h->fork_ev) cudaEventDestroy(h->fork_ev);
    if (h->cap_stream) cudaStreamDestroy(h->cap_stream);
    void* const blocks[] = {h->buf[0], h->buf[1], h->varpi, h->u_prev, h->partials, h->out8};
    for (void* p : blocks)
        if (p && (!h->pooled || cudaFreeAsync(p, h->stream) != cudaSuccess)) cudaFree(p);
    cudaFree(h->varpi3);
    cudaFree(h->links);
    if (h->pool) cudaStreamSynchronize(h->stream);  // the pool may serve another stream next
    slot_release(h->out8_host);
    pool_release(h->pool);
}

// One direct time step on `s`, updating the bookkeeping.
int step_once(hlbm_t* h, cudaStream_t s) {
    const LaunchCtx c = h->ctx(s);
    if (h->pattern == HLBM_TWO_LATTICE) {
        HLBM_CUDA(launch_step(c, MODE_TWO_LATTICE, h->buf[h->cur], h->buf[1 - h->cur], h->varpi));
        h->cur = 1 - h->cur;
    } else {
        HLBM_CUDA(launch_step(c, h->aa_odd ? MODE_AA_ODD : MODE_AA_EVEN, h->buf[0], h->buf[0], h->varpi));
        h->aa_odd = 1 - h->aa_odd;
    }
    return HLBM_OK;
}

bool resident(const hlbm_t* h, long n) {
    return h->pattern == HLBM_TWO_LATTICE && n >= kResidentMin && resident_applies(h->ctx(h->stream));
}
bool two_steps(const hlbm_t* h) { return h->pattern == HLBM_TWO_LATTICE && step2_applies(h->ctx(h->stream)); }

// n steps on `s`, where `two` in pairs of two-step launches: four steps then end in the buffer
// that they began in, as single steps do (a caller may capture them and replay the graph).
int steps_on(hlbm_t* h, cudaStream_t s, long n, bool two) {
    int rc = HLBM_OK;
    for (; two && n >= 4; n -= 4) {
        HLBM_CUDA(launch_step2(h->ctx(s), h->buf[h->cur], h->buf[1 - h->cur], h->varpi));
        HLBM_CUDA(launch_step2(h->ctx(s), h->buf[1 - h->cur], h->buf[h->cur], h->varpi));
    }
    for (; n > 0 && rc == HLBM_OK; --n) rc = step_once(h, s);
    return rc;
}

bool at_graph_origin(const hlbm_t* h) { return h->pattern == HLBM_TWO_LATTICE ? h->cur == 0 : h->aa_odd == 0; }

// Capture what `body` launches on the handle's capture stream, starting from the graph origin layout,
// which an even number of steps returns to.
template <class Body>
int capture(hlbm_t* h, cudaGraphExec_t* exec, Body&& body) {
    if (!h->cap_stream) HLBM_CUDA(cudaStreamCreateWithFlags(&h->cap_stream, cudaStreamNonBlocking));
    const int cur0 = h->cur, odd0 = h->aa_odd;
    cudaGraph_t graph = nullptr;
    HLBM_CUDA(cudaStreamBeginCapture(h->cap_stream, cudaStreamCaptureModeThreadLocal));
    const int rc = body(h->cap_stream);
    cudaError_t e = cudaStreamEndCapture(h->cap_stream, &graph);
    h->cur = cur0;
    h->aa_odd = odd0;
    if (rc != HLBM_OK) {
        if (graph) cudaGraphDestroy(graph);
        return rc;
    }
    if (e != cudaSuccess) return cuda_fail(e);
    if (*exec) {
        cudaGraphExecDestroy(*exec);
        *exec = nullptr;
    }
    e = cudaGraphInstantiate(exec, graph, 0);
    cudaGraphDestroy(graph);
    return e == cudaSuccess ? HLBM_OK : cuda_fail(e);
}

// Step graph k. In place (AA) a kernel overwrites what it reads, so its successor must not start
// early: the caches of an SM may hold values from before the overwriting.
int build_graph(hlbm_t* h, int k) {
    const bool two = two_steps(h);
    const int rc = capture(h, &h->gexec[k], [h, k, two](cudaStream_t s) {
        if (two) return steps_on(h, s, kGraphSteps[k], true);
        const int r = step_once(h, s);  // launched plainly: it follows whatever came before the graph
        if (h->pattern == HLBM_TWO_LATTICE) h->chaining = CHAIN_GRAPH;
        return r == HLBM_OK ? steps_on(h, s, kGraphSteps[k] - 1, false) : r;
    });
    h->chaining = CHAIN_NONE;
    h->graph_valid[k] = rc == HLBM_OK;
    return rc;
}

// kSeriesSamples times `every` steps and the diagnostics, into the records behind out8. The
// diagnostics of a sample run beside the steps that follow it, up to the one that overwrites
// the state they read (in place, that is the next one).
int build_series(hlbm_t* h, int every) {
    if (!h->series_stream) HLBM_CUDA(cudaStreamCreateWithFlags(&h->series_stream, cudaStreamNonBlocking));
    for (cudaEvent_t& e : h->series_ev)
        if (!e) HLBM_CUDA(cudaEventCreateWithFlags(&e, cudaEventDisableTiming));
    const int rc = capture(h, &h->series_exec, [h, every](cudaStream_t s) {
        const bool in_place = h->pattern != HLBM_TWO_LATTICE;
        cudaStream_t d = h->series_stream;
        bool read[2] = {};  // by diagnostics that the steps have not waited for
        for (int k = 0; k < kSeriesSamples; ++k) {
            for (int j = 0; j < every; ++j) {
                const int to = in_place ? 0 : 1 - h->cur;
                if (read[to]) HLBM_CUDA(cudaStreamWaitEvent(s, h->series_ev[to], 0));
                read[to] = false;
                const int r = step_once(h, s);
                if (r != HLBM_OK) return r;
            }
            HLBM_CUDA(cudaEventRecord(h->series_ev[2], s));
            HLBM_CUDA(cudaStreamWaitEvent(d, h->series_ev[2], 0));
            HLBM_CUDA(launch_reduce(h->ctx(d), h->layout(), h->state(), h->u_prev, 0, h->partials, h->out8 + 8 * (k + 1)));
            const int from = in_place ? 0 : h->cur;
            HLBM_CUDA(cudaEventRecord(h->series_ev[from], d));
            read[from] = true;
        }
        for (int b = 0; b < 2; ++b)
            if (read[b]) HLBM_CUDA(cudaStreamWaitEvent(s, h->series_ev[b], 0));
        return (int)HLBM_OK;
    });
    if (rc == HLBM_OK) h->series_every = every;
    return rc;
}

int reset_counters(hlbm_t* h) {
    h->step = 0;
    HLBM_CUDA(cudaMemsetAsync(h->u_prev, 0, 3 * h->cells * h->arith_bytes(), h->stream));
    return HLBM_OK;
}

// The solid cells rest in every buffer: steps leave them alone, so they would otherwise hold what
// the memory held before, and show it in a checkpoint or once the mask is removed.
cudaError_t rest_solids(hlbm_t* h) {
    cudaError_t e = cudaSuccess;
    for (void* b : h->buf)
        if (b && h->links && e == cudaSuccess) e = launch_rest_solid(h->ctx(h->stream), b);
    return e;
}

// Write natural FP64 populations (device pointer; q values if uniform) as the new state.
int write_state(hlbm_t* h, const double* fnat_dev, int uniform) {
    h->cur = 0;
    h->aa_odd = 0;
    const int lay = h->layout();
    HLBM_CUDA(launch_write_state(h->ctx(h->stream), lay, fnat_dev, uniform, h->buf[0]));
    return reset_counters(h);
}

bool is_finite(double v) { return std::isfinite(v); }

// Host-side equilibrium at (rho0, u0) in the documented direction order
// (the same second-order expansion the kernels use, evaluated once).
void host_equilibrium(int q, double rho, const double u[3], double* out) {
    static const int c9[9][3] = {{0, 0, 0}, {1, 0, 0}, {0, 1, 0}, {-1, 0, 0}, {0, -1, 0},
                                 {1, 1, 0}, {-1, 1, 0}, {-1, -1, 0}, {1, -1, 0}};
    static const int c19[19][3] = {{0, 0, 0},  {1, 0, 0},   {-1, 0, 0}, {0, 1, 0},  {0, -1, 0},
                                   {0, 0, 1},  {0, 0, -1},  {1, 1, 0},  {-1, -1, 0}, {1, -1, 0},
                                   {-1, 1, 0}, {1, 0, 1},   {-1, 0, -1}, {1, 0, -1}, {-1, 0, 1},
                                   {0, 1, 1},  {0, -1, -1}, {0, 1, -1}, {0, -1, 1}};
    const double uu = u[0] * u[0] + u[1] * u[1] + u[2] * u[2];
    for (int i = 0; i < q; ++i) {
        const int* c = q == 9 ? c9[i] : c19[i];
        const int c2 = c[0] * c[0] + c[1] * c[1] + c[2] * c[2];
        const double w = q == 9 ? (c2 == 0 ? 4.0 / 9 : (c2 == 1 ? 1.0 / 9 : 1.0 / 36))
                                : (c2 == 0 ? 1.0 / 3 : (c2 == 1 ? 1.0 / 18 : 1.0 / 36));
        const double cu = c[0] * u[0] + c[1] * u[1] + c[2] * u[2];
        out[i] = w * rho * (1.0 + 3.0 * cu + 4.5 * cu * cu - 1.5 * uu);
    }
}

struct CkptHeader {
    char magic[8];
    int q, nx, ny, nz, storage, pattern, cur, aa_odd;
    long long step;
    double tau, F[3], scale;
    int bc[3], pad;
};

}  // namespace

extern "C" {

const char* hlbm_strerror(int status) {
    switch (status) {
        case HLBM_OK: return "ok";
        case HLBM_ERR_INVALID_ARG: return "invalid argument";
        case HLBM_ERR_OOM: return "out of memory";
        case HLBM_ERR_CUDA: return "CUDA error";
        case HLBM_ERR_NOT_CONVERGED: return "not converged";
        case HLBM_ERR_TIMEOUT: return "timeout";
        case HLBM_ERR_BUSY: return "busy";
        case HLBM_ERR_IO: return "I/O error";
        case HLBM_ERR_STATE: return "invalid state for this call";
        case HLBM_ERR_CANCELLED: return "cancelled";
        case HLBM_ERR_SCRATCH_LIMIT: return "lattice too large for the fixed scratch of the allocation-free call";
    }
    return "unknown status";
}

const char* hlbm_last_cuda_error(void) { return g_last_cuda; }

int hlbm_create(hlbm_t** out, int velset, int nx, int ny, int nz, int storage, int pattern, void* cuda_stream) {
    if (!out) return HLBM_ERR_INVALID_ARG;
    *out = nullptr;
    if (velset != HLBM_D2Q9 && velset != HLBM_D3Q19) return HLBM_ERR_INVALID_ARG;
    if (nx < 1 || ny < 1 || nz < 1) return HLBM_ERR_INVALID_ARG;
    if (velset == HLBM_D2Q9 && nz != 1) return HLBM_ERR_INVALID_ARG;
    if (storage < HLBM_F64 || storage > HLBM_BF16DEV) return HLBM_ERR_INVALID_ARG;
    if (pattern != HLBM_TWO_LATTICE && pattern != HLBM_AA) return HLBM_ERR_INVALID_ARG;
    if (ny > 65535 || nz > 65535) return HLBM_ERR_INVALID_ARG;  // launch-grid y and z limits
    const size_t cells = (size_t)nx * ny * nz;
    if (cells > ((size_t)1 << 34)) return HLBM_ERR_INVALID_ARG;

    hlbm_t* h = new (std::nothrow) hlbm_lattice();
    if (!h) return HLBM_ERR_OOM;
    h->q = velset;
    h->nx = nx;
    h->ny = ny;
    h->nz = nz;
    h->storage = storage;
    h->pattern = pattern;
    h->cells = cells;
    h->stream = static_cast<cudaStream_t>(cuda_stream);
    h->scale = storage == HLBM_F16DEV ? 4096.0 : 1.0;
    cudaError_t e = cudaGetDevice(&h->device);
    const size_t nparts = reduce_partials_count(h->ctx(h->stream));
    h->pooled = pool_keeps((pattern == HLBM_TWO_LATTICE ? 2 : 1) * h->state_bytes() + cells * (sizeof(float) + 3 * h->arith_bytes()));
    if (e == cudaSuccess) e = lattice_alloc(h, (void**)&h->buf[0], h->state_bytes());
    if (e == cudaSuccess && pattern == HLBM_TWO_LATTICE) e = lattice_alloc(h, (void**)&h->buf[1], h->state_bytes());
    if (e == cudaSuccess) e = lattice_alloc(h, (void**)&h->varpi, cells * sizeof(float));
    if (e == cudaSuccess) e = lattice_alloc(h, (void**)&h->u_prev, 3 * cells * h->arith_bytes());
    if (e == cudaSuccess) e = lattice_alloc(h, (void**)&h->partials, nparts * 8 * sizeof(double));
    if (e == cudaSuccess) e = lattice_alloc(h, (void**)&h->out8, (1 + kSeriesSamples) * 8 * sizeof(double));
    if (e == cudaSuccess && !(h->out8_host = slot_acquire())) e = cudaErrorMemoryAllocation;
    if (e == cudaSuccess) e = launch_fill_f32(h->varpi, cells, 1.0f, h->stream);
    if (e != cudaSuccess) {
        int rc = cuda_fail(e);
        free_all(h);
        delete h;
        return rc;
    }
    int rc = hlbm_init_equilibrium(h, 1.0, 0.0, 0.0, 0.0);
    if (rc == HLBM_OK) {
        cudaError_t s = cudaStreamSynchronize(h->stream);
        if (s != cudaSuccess) rc = cuda_fail(s);
    }
    if (rc != HLBM_OK) {
        free_all(h);
        delete h;
        return rc;
    }
    *out = h;
    return HLBM_OK;
}

void hlbm_destroy(hlbm_t* h) {
    if (!h) return;
    DeviceGuard g(h->device);
    if (h->moved) cudaDeviceSynchronize();
    else cudaStreamSynchronize(h->stream);
    free_all(h);
    delete h;
}

int hlbm_release_scratch(hlbm_t* h) {
    if (!h) return HLBM_ERR_INVALID_ARG;
    DeviceGuard g(h->device);
    HLBM_CUDA(cudaStreamSynchronize(h->stream));
    if (h->pool) HLBM_CUDA(cudaMemPoolTrimTo(h->pool, 0));
    memory_give_back();
    return HLBM_OK;
}

int hlbm_set_stream(hlbm_t* h, void* cuda_stream) {
    if (!h) return HLBM_ERR_INVALID_ARG;
    h->moved = h->moved || h->stream != static_cast<cudaStream_t>(cuda_stream);
    h->stream = static_cast<cudaStream_t>(cuda_stream);
    return HLBM_OK;
}

int hlbm_set_relaxation(hlbm_t* h, double tau) {
    if (!h || !is_finite(tau) || !(tau > 0.5)) return HLBM_ERR_INVALID_ARG;
    h->tau = tau;
    h->settings_changed();
    return HLBM_OK;
}

int hlbm_set_force(hlbm_t* h, double Fx, double Fy, double Fz) {
    if (!h || !is_finite(Fx) || !is_finite(Fy) || !is_finite(Fz)) return HLBM_ERR_INVALID_ARG;
    h->F[0] = Fx;
    h->F[1] = Fy;
    h->F[2] = h->q == HLBM_D2Q9 ? 0.0 : Fz;
    h->settings_changed();
    return HLBM_OK;
}

int hlbm_set_boundary(hlbm_t* h, int axis, int type) {
    if (!h || axis < 0 || axis > 2) return HLBM_ERR_INVALID_ARG;
    if (type != HLBM_PERIODIC && type != HLBM_HALFWAY_BOUNCE_BACK) return HLBM_ERR_INVALID_ARG;
    if (h->q == HLBM_D2Q9 && axis == 2 && type != HLBM_PERIODIC) return HLBM_ERR_INVALID_ARG;
    if (h->bc[axis] == type) return HLBM_OK;
    if (h->links) return HLBM_ERR_STATE;  // set boundaries before the solid mask
    if (h->pattern == HLBM_AA) {
        // The AA layouts place bounced populations according to the walls:
        // re-lay the post-collision state under the new boundary.
        DeviceGuard g(h->device);
        double* tmp = nullptr;
        HLBM_CUDA(scratch_alloc(h, (void**)&tmp, (size_t)h->q * h->cells * sizeof(double)));
        cudaError_t e = launch_read_state(h->ctx(h->stream), h->layout(), h->state(), tmp);
        h->bc[axis] = type;
        if (e == cudaSuccess) e = launch_write_state(h->ctx(h->stream), h->layout(), tmp, 0, h->buf[0]);
        cudaFreeAsync(tmp, h->stream);
        if (e != cudaSuccess) return cuda_fail(e);
    }
    h->bc[axis] = type;
    h->settings_changed();
    return HLBM_OK;
}

int hlbm_set_homogenization(hlbm_t* h, int form) {
    if (!h || (form != HLBM_HOMOG_SHIFT && form != HLBM_HOMOG_DRAG)) return HLBM_ERR_INVALID_ARG;
    if (form == HLBM_HOMOG_DRAG && h->aniso) return HLBM_ERR_STATE;  // the tensor form is a shift form
    h->homog = form;
    h->settings_changed();
    return HLBM_OK;
}

int hlbm_set_step_kernel(hlbm_t* h, int variant) {
    if (!h || (variant != HLBM_STEP_AUTO && variant != HLBM_STEP_PER_CELL)) return HLBM_ERR_INVALID_ARG;
    h->step_variant = variant;
    h->settings_changed();
    return HLBM_OK;
}

int hlbm_set_storage_scale(hlbm_t* h, double s) {
    if (!h || !is_finite(s)) return HLBM_ERR_INVALID_ARG;
    if (h->storage != HLBM_F16DEV) return s == 1.0 ? HLBM_OK : HLBM_ERR_INVALID_ARG;
    int ex = 0;
    const double m = std::frexp(s, &ex);
    if (m != 0.5 || s < 1.0 || s > 1048576.0) return HLBM_ERR_INVALID_ARG;
    h->scale = s;
    h->settings_changed();
    return HLBM_OK;
}

int hlbm_porosity_from_permeability(const float* K, double nu, double tau, float* varpi, size_t n) {
    if ((!K || !varpi) && n) return HLBM_ERR_INVALID_ARG;
    if (!is_finite(nu) || !is_finite(tau) || nu <= 0.0 || tau <= 0.0) return HLBM_ERR_INVALID_ARG;
    for (size_t k = 0; k < n; ++k) {
        const double Kk = K[k];
        double v = Kk > 0.0 ? 1.0 - nu * tau / Kk : 0.0;  // NaN and K <= 0 give 0
        if (!(v >= 0.0)) v = 0.0;
        if (v > 1.0) v = 1.0;
        varpi[k] = (float)v;
    }
    return HLBM_OK;
}

// The handle returns to the scalar porosity field; the captured step graph
// only needs rebuilding when the tensor form was in use (the field's device
// buffer itself does not move).
static void use_scalar_porosity(hlbm_t* h) {
    if (h->aniso) {
        h->aniso = 0;
        h->settings_changed();
    }
}

// Check a device array of n porosity values and copy it into the handle's
// field; the field is unchanged when a value is rejected. Synchronises.
static int porosity_from_device(hlbm_t* h, const float* varpi, size_t n) {
    int* bad = nullptr;
    HLBM_CUDA(scratch_alloc(h, (void**)&bad, sizeof(int)));
    int nbad = 0;
    cudaError_t e = cudaMemsetAsync(bad, 0, sizeof(int), h->stream);
    if (e == cudaSuccess) e = launch_check_unit_interval(varpi, n, bad, h->stream);
    if (e == cudaSuccess) e = cudaMemcpyAsync(&nbad, bad, sizeof(int), cudaMemcpyDeviceToHost, h->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(h->stream);
    cudaFreeAsync(bad, h->stream);
    if (e != cudaSuccess) return cuda_fail(e);
    if (nbad) return HLBM_ERR_INVALID_ARG;
    HLBM_CUDA(cudaMemcpyAsync(h->varpi, varpi, n * sizeof(float), cudaMemcpyDeviceToDevice, h->stream));
    use_scalar_porosity(h);
    return HLBM_OK;
}

int hlbm_set_porosity(hlbm_t* h, const float* varpi, int on_device) {
    if (!h || !varpi) return HLBM_ERR_INVALID_ARG;
    DeviceGuard g(h->device);
    const size_t n = h->cells;
    if (on_device) return porosity_from_device(h, varpi, n);
    // A host array goes to a device staging buffer and is checked there (a
    // single host core reads the 64 MiB of a 256^3 field far slower than the
    // copy and a check kernel take); without room for the staging buffer it is
    // checked on the host and copied straight into the field.
    float* stage = nullptr;
    if (scratch_alloc(h, (void**)&stage, n * sizeof(float)) != cudaSuccess) {
        (void)cudaGetLastError();  // the failed allocation leaves no sticky error
        if (!host_unit_interval(varpi, n)) return HLBM_ERR_INVALID_ARG;
        HLBM_CUDA(cudaMemcpyAsync(h->varpi, varpi, n * sizeof(float), cudaMemcpyHostToDevice, h->stream));
        HLBM_CUDA(cudaStreamSynchronize(h->stream));
        use_scalar_porosity(h);
        return HLBM_OK;
    }
    cudaError_t e = cudaMemcpyAsync(stage, varpi, n * sizeof(float), cudaMemcpyHostToDevice, h->stream);
    const int rc = e == cudaSuccess ? porosity_from_device(h, stage, n) : cuda_fail(e);
    cudaFreeAsync(stage, h->stream);
    if (rc != HLBM_OK) cudaStreamSynchronize(h->stream);  // the host array may be reused at once
    return rc;
}

int hlbm_set_solid_mask(hlbm_t* h, const unsigned char* solid, int on_device) {
    if (!h) return HLBM_ERR_INVALID_ARG;
    DeviceGuard g(h->device);
    if (!solid) {  // remove the obstacles
        if (h->links) {
            // in place, populations that bounced off a solid cell lie elsewhere than ones that
            // travelled on: re-lay the state (two lattices hold it unstreamed)
            double* nat = nullptr;
            if (h->pattern != HLBM_TWO_LATTICE) HLBM_CUDA(scratch_alloc(h, (void**)&nat, (size_t)h->q * h->cells * sizeof(double)));
            LaunchCtx c = h->ctx(h->stream);
            cudaError_t e = nat ? launch_read_state(c, h->layout(), h->state(), nat) : cudaSuccess;
            c.links = nullptr;
            if (nat && e == cudaSuccess) e = launch_write_state(c, h->layout(), nat, 0, h->state());
            if (nat) cudaFreeAsync(nat, h->stream);
            if (e == cudaSuccess) e = cudaStreamSynchronize(h->stream);
            if (e != cudaSuccess) return cuda_fail(e);
            cudaFree(h->links);
            h->links = nullptr;
        }
        h->settings_changed();
        return HLBM_OK;
    }
    // the state's layout (AA) depends on the obstacles: keep the post-collision
    // state across the change, as hlbm_set_boundary does
    double* tmp = nullptr;
    unsigned char* dsolid = nullptr;
    HLBM_CUDA(scratch_alloc(h, (void**)&tmp, (size_t)h->q * h->cells * sizeof(double)));
    cudaError_t e = launch_read_state(h->ctx(h->stream), h->layout(), h->state(), tmp);
    if (e == cudaSuccess && !h->links) e = device_malloc((void**)&h->links, h->cells * sizeof(unsigned));
    if (e == cudaSuccess && !on_device) e = scratch_alloc(h, (void**)&dsolid, h->cells);
    if (e == cudaSuccess && !on_device) e = cudaMemcpyAsync(dsolid, solid, h->cells, cudaMemcpyHostToDevice, h->stream);
    if (e == cudaSuccess) e = launch_build_links(h->ctx(h->stream), on_device ? solid : dsolid, h->links);
    if (e == cudaSuccess) e = launch_write_state(h->ctx(h->stream), h->layout(), tmp, 0, h->state());
    if (e == cudaSuccess) e = rest_solids(h);
    if (dsolid) cudaFreeAsync(dsolid, h->stream);
    cudaFreeAsync(tmp, h->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(h->stream);
    if (e != cudaSuccess) return cuda_fail(e);
    h->settings_changed();
    return HLBM_OK;
}

int hlbm_set_porosity_tensor(hlbm_t* h, const float* varpi3, int on_device) {
    if (!h || !varpi3) return HLBM_ERR_INVALID_ARG;
    if (h->homog != HLBM_HOMOG_SHIFT) return HLBM_ERR_STATE;
    DeviceGuard g(h->device);
    const size_t n = 3 * h->cells;
    if (!h->varpi3) HLBM_CUDA(device_malloc((void**)&h->varpi3, n * sizeof(float)));
    if (!on_device) {
        if (!host_unit_interval(varpi3, n)) return HLBM_ERR_INVALID_ARG;
        HLBM_CUDA(cudaMemcpyAsync(h->varpi3, varpi3, n * sizeof(float), cudaMemcpyHostToDevice, h->stream));
        HLBM_CUDA(cudaStreamSynchronize(h->stream));
    } else {
        int* bad = nullptr;
        HLBM_CUDA(scratch_alloc(h, (void**)&bad, sizeof(int)));
        int nbad = 0;
        cudaError_t e = cudaMemsetAsync(bad, 0, sizeof(int), h->stream);
        if (e == cudaSuccess) e = launch_check_unit_interval(varpi3, n, bad, h->stream);
        if (e == cudaSuccess) e = cudaMemcpyAsync(&nbad, bad, sizeof(int), cudaMemcpyDeviceToHost, h->stream);
        if (e == cudaSuccess) e = cudaStreamSynchronize(h->stream);
        cudaFreeAsync(bad, h->stream);
        if (e != cudaSuccess) return cuda_fail(e);
        if (nbad) return HLBM_ERR_INVALID_ARG;
        HLBM_CUDA(cudaMemcpyAsync(h->varpi3, varpi3, n * sizeof(float), cudaMemcpyDeviceToDevice, h->stream));
    }
    h->aniso = 1;
    h->settings_changed();
    return HLBM_OK;
}

int hlbm_init_equilibrium(hlbm_t* h, double rho0, double ux, double uy, double uz) {
    if (!h || !is_finite(rho0) || !is_finite(ux) || !is_finite(uy) || !is_finite(uz) || !(rho0 > 0.0))
        return HLBM_ERR_INVALID_ARG;
    DeviceGuard g(h->device);
    double u[3] = {ux, uy, h->q == HLBM_D2Q9 ? 0.0 : uz};
    double feq[19];
    host_equilibrium(h->q, rho0, u, feq);
    double* dev = nullptr;
    HLBM_CUDA(scratch_alloc(h, (void**)&dev, sizeof(feq)));
    cudaError_t e = cudaMemcpyAsync(dev, feq, h->q * sizeof(double), cudaMemcpyHostToDevice, h->stream);
    int rc = e == cudaSuccess ? write_state(h, dev, 1) : cuda_fail(e);
    // the pageable source above is consumed before cudaMemcpyAsync returns
    cudaFreeAsync(dev, h->stream);
    return rc;
}

int hlbm_set_populations(hlbm_t* h, const double* f, int on_device) {
    if (!h || !f) return HLBM_ERR_INVALID_ARG;
    DeviceGuard g(h->device);
    const size_t bytes = (size_t)h->q * h->cells * sizeof(double);
    if (on_device) return write_state(h, f, 0);
    double* dev = nullptr;
    HLBM_CUDA(scratch_alloc(h, (void**)&dev, bytes));
    cudaError_t e = cudaMemcpyAsync(dev, f, bytes, cudaMemcpyHostToDevice, h->stream);
    int rc = e == cudaSuccess ? write_state(h, dev, 0) : cuda_fail(e);
    cudaFreeAsync(dev, h->stream);
    if (rc == HLBM_OK) {
        e = cudaStreamSynchronize(h->stream);
        if (e != cudaSuccess) rc = cuda_fail(e);
    }
    return rc;
}

int hlbm_get_populations(hlbm_t* h, double* f, int on_device) {
    if (!h || !f) return HLBM_ERR_INVALID_ARG;
    DeviceGuard g(h->device);
    const LaunchCtx c = h->ctx(h->stream);
    if (on_device) {
        HLBM_CUDA(launch_read_state(c, h->layout(), h->state(), f));
        return HLBM_OK;
    }
    const size_t bytes = (size_t)h->q * h->cells * sizeof(double);
    double* dev = nullptr;
    HLBM_CUDA(scratch_alloc(h, (void**)&dev, bytes));
    cudaError_t e = launch_read_state(c, h->layout(), h->state(), dev);
    if (e == cudaSuccess) e = cudaMemcpyAsync(f, dev, bytes, cudaMemcpyDeviceToHost, h->stream);
    cudaFreeAsync(dev, h->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(h->stream);
    return e == cudaSuccess ? HLBM_OK : cuda_fail(e);
}

int hlbm_step(hlbm_t* h, long nsteps) {
    if (!h || nsteps < 0) return HLBM_ERR_INVALID_ARG;
    DeviceGuard g(h->device);
    long left = nsteps;
    if (resident(h, left)) {
        while (left >= kResidentMin) {
            const long n = left < kResidentMax ? left : kResidentMax;
            HLBM_CUDA(launch_resident(h->ctx(h->stream), h->state(), h->varpi, (int)n));
            left -= n;
            h->step += n;
        }
    }
    const bool two = left >= 4 && two_steps(h);
    h->graph_steps += left;
    const bool use_long = h->graph_valid[1] || h->graph_steps >= kLongFrom;
    while (left > 0) {
        const int k = use_long && left >= kGraphSteps[1];
        const bool use = k || h->graph_valid[0] || !h->graph_valid[1] || h->graph_steps >= kShortFrom;
        if (use && left >= kGraphSteps[0] && at_graph_origin(h)) {
            if (!h->graph_valid[k]) {
                int rc = build_graph(h, k);
                if (rc != HLBM_OK) return rc;
            }
            HLBM_CUDA(cudaGraphLaunch(h->gexec[k], h->stream));
            left -= kGraphSteps[k];
            h->step += kGraphSteps[k];
        } else {
            const int n = two && left >= 4 && (!use || left < kGraphSteps[0]) ? 4 : 1;
            int rc = steps_on(h, h->stream, n, two);
            if (rc != HLBM_OK) return rc;
            left -= n;
            h->step += n;
        }
    }
    return HLBM_OK;
}

int hlbm_steps_per_launch(hlbm_t* h, long nsteps, long* steps) {
    if (!h || !steps || nsteps < 0) return HLBM_ERR_INVALID_ARG;
    DeviceGuard g(h->device);
    if (resident(h, nsteps)) *steps = nsteps < kResidentMax ? nsteps : kResidentMax;
    else *steps = nsteps >= 4 && two_steps(h) ? 2 : 1;
    return HLBM_OK;
}

int hlbm_get_step(hlbm_t* h, long long* step) {
    if (!h || !step) return HLBM_ERR_INVALID_ARG;
    *step = h->step;
    return HLBM_OK;
}

static int moments_common(hlbm_t* h, void* rho, void* u, int on_device, int f64) {
    if (!h) return HLBM_ERR_INVALID_ARG;
    if (!rho && !u) return HLBM_OK;
    DeviceGuard g(h->device);
    const LaunchCtx c = h->ctx(h->stream);
    if (on_device) {
        HLBM_CUDA(launch_moments(c, h->layout(), h->state(), rho, u, f64));
        return HLBM_OK;
    }
    const size_t es = f64 ? 8 : 4;
    void* drho = nullptr;
    void* du = nullptr;
    cudaError_t e = cudaSuccess;
    if (rho) e = scratch_alloc(h, (void**)&drho, h->cells * es);
    if (e == cudaSuccess && u) e = scratch_alloc(h, (void**)&du, 3 * h->cells * es);
    if (e == cudaSuccess) e = launch_moments(c, h->layout(), h->state(), drho, du, f64);
    if (e == cudaSuccess && rho) e = cudaMemcpyAsync(rho, drho, h->cells * es, cudaMemcpyDeviceToHost, h->stream);
    if (e == cudaSuccess && u) e = cudaMemcpyAsync(u, du, 3 * h->cells * es, cudaMemcpyDeviceToHost, h->stream);
    if (drho) cudaFreeAsync(drho, h->stream);
    if (du) cudaFreeAsync(du, h->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(h->stream);
    return e == cudaSuccess ? HLBM_OK : cuda_fail(e);
}

int hlbm_moments(hlbm_t* h, float* rho, float* u, int on_device) { return moments_common(h, rho, u, on_device, 0); }

int hlbm_moments_f64(hlbm_t* h, double* rho, double* u, int on_device) {
    return moments_common(h, rho, u, on_device, 1);
}

int hlbm_reduce(hlbm_t* h, hlbm_stats* out) {
    if (!h || !out) return HLBM_ERR_INVALID_ARG;
    DeviceGuard g(h->device);
    HLBM_CUDA(launch_reduce(h->ctx(h->stream), h->layout(), h->state(), h->u_prev, 1, h->partials, h->out8));
    HLBM_CUDA(cudaMemcpyAsync(h->out8_host, h->out8, 8 * sizeof(double), cudaMemcpyDeviceToHost, h->stream));
    HLBM_CUDA(cudaStreamSynchronize(h->stream));
    const double* v = h->out8_host;
    out->mass = v[0];
    out->momentum[0] = v[1];
    out->momentum[1] = v[2];
    out->momentum[2] = v[3];
    out->plane_flux = v[4];
    out->k_app = v[5];
    out->max_du = v[6];
    out->max_u = v[7];
    out->step = h->step;
    return HLBM_OK;
}

int hlbm_reduce_series(hlbm_t* h, long nsamples, int every, double* out, int on_device) {
    if (!h || !out || nsamples < 1 || every < 1) return HLBM_ERR_INVALID_ARG;
    DeviceGuard g(h->device);
    const size_t bytes = (size_t)nsamples * 8 * sizeof(double);
    double* dst = out;
    if (!on_device) HLBM_CUDA(scratch_alloc(h, (void**)&dst, bytes));
    int rc = HLBM_OK;
    cudaStreamCaptureStatus capturing = cudaStreamCaptureStatusNone;
    // (runs of four and more steps go two per launch where that applies, which gains more than the
    // graph: 160^3, 63 samples every 4 steps, 30.3 ms replayed, 28.8 ms launched)
    bool graphs = every < kResidentMin && nsamples >= kSeriesMin && !(every >= 4 && two_steps(h));
    if (graphs && (cudaStreamIsCapturing(h->stream, &capturing) != cudaSuccess || capturing != cudaStreamCaptureStatusNone)) {
        (void)cudaGetLastError();
        graphs = false;  // a caller's capture takes the single launches
    }
    for (long k = 0; k < nsamples && rc == HLBM_OK;) {
        if (graphs && k && nsamples - k >= kSeriesSamples && at_graph_origin(h)) {
            if (h->series_every != every) rc = build_series(h, every);
            if (rc != HLBM_OK) break;
            cudaError_t e = cudaGraphLaunch(h->series_exec, h->stream);
            if (e == cudaSuccess)
                e = cudaMemcpyAsync(dst + 8 * k, h->out8 + 8, kSeriesSamples * 8 * sizeof(double), cudaMemcpyDeviceToDevice,
                                    h->stream);
            if (e != cudaSuccess) rc = cuda_fail(e);
            h->step += (long long)kSeriesSamples * every;
            k += kSeriesSamples;
            continue;
        }
        if (k) rc = hlbm_step(h, every);
        if (rc == HLBM_OK) {
            const cudaError_t e = launch_reduce(h->ctx(h->stream), h->layout(), h->state(), h->u_prev, 0,
                                                h->partials, dst + 8 * k);
            if (e != cudaSuccess) rc = cuda_fail(e);
        }
        ++k;
    }
    if (!on_device) {
        cudaError_t e = cudaSuccess;
        if (rc == HLBM_OK) e = cudaMemcpyAsync(out, dst, bytes, cudaMemcpyDeviceToHost, h->stream);
        const cudaError_t ef = cudaFreeAsync(dst, h->stream);
        if (e == cudaSuccess) e = ef;
        if (e == cudaSuccess) e = cudaStreamSynchronize(h->stream);
        if (rc == HLBM_OK && e != cudaSuccess) rc = cuda_fail(e);
    }
    return rc;
}

namespace {

// Device allocations of one call, released on every exit path (stream-ordered).
struct Scratch {
    hlbm_t* h;
    std::vector<void*> ptrs;
    explicit Scratch(hlbm_t* hh) : h(hh) {}
    ~Scratch() {
        for (void* p : ptrs) cudaFreeAsync(p, h->stream);
    }
    cudaError_t alloc(void** p, size_t bytes) {
        cudaError_t e = scratch_alloc(h, p, bytes);
        if (e == cudaSuccess) ptrs.push_back(*p);
        return e;
    }
};

// A stream for the length of a call, behind what the handle's stream holds so far. Chained kernels
// (launch_chained) must follow one another directly: on the caller's stream another thread, with
// a handle of its own, can put a copy or a graph between two of them, and here nobody can.
// Waited for at the latest when the call ends, before its scratch is given back.
struct OwnStream {
    cudaStream_t s = nullptr;
    ~OwnStream() {
        if (s) stream_release(s, cudaStreamSynchronize(s) == cudaSuccess);
    }
    cudaError_t fork(hlbm_t* h) {
        cudaError_t e = stream_acquire(&s);
        if (e == cudaSuccess && !h->fork_ev) e = cudaEventCreateWithFlags(&h->fork_ev, cudaEventDisableTiming);
        if (e == cudaSuccess) e = cudaEventRecord(h->fork_ev, h->stream);
        return e == cudaSuccess ? cudaStreamWaitEvent(s, h->fork_ev, 0) : e;
    }
};

// Copy the current state into `dst` in the NATURAL layout, on c's stream. tmp: q doubles per
// cell, for the in-place pattern.
int copy_natural(hlbm_t* h, const LaunchCtx& c, void* dst, double* tmp) {
    if (h->pattern == HLBM_TWO_LATTICE) {
        HLBM_CUDA(cudaMemcpyAsync(dst, h->state(), h->state_bytes(), cudaMemcpyDeviceToDevice, c.stream));
        return HLBM_OK;
    }
    HLBM_CUDA(launch_read_state(c, h->layout(), h->state(), tmp));
    HLBM_CUDA(launch_write_state(c, kNatural, tmp, 0, dst));
    return HLBM_OK;
}

// Make a NATURAL-layout buffer the handle's state, on c's stream.
int adopt_natural(hlbm_t* h, const LaunchCtx& c, const void* src, double* tmp) {
    if (h->pattern == HLBM_TWO_LATTICE) {
        HLBM_CUDA(cudaMemcpyAsync(h->buf[0], src, h->state_bytes(), cudaMemcpyDeviceToDevice, c.stream));
        h->cur = 0;
        return HLBM_OK;
    }
    HLBM_CUDA(launch_read_state(c, kNatural, src, tmp));
    h->aa_odd = 0;
    HLBM_CUDA(launch_write_state(c, h->layout(), tmp, 0, h->buf[0]));
    return HLBM_OK;
}

}  // namespace

int hlbm_adjoint_flux_grad(hlbm_t* h, long nsteps, int every, int plane_x, double* J, float* grad, int on_device) {
    if (!h || !J || !grad || nsteps < 0 || every < 1 || plane_x < 0 || plane_x >= (h ? h->nx : 0))
        return HLBM_ERR_INVALID_ARG;
    // the adjoint differentiates the isotropic shift form without obstacles
    if (h->homog != HLBM_HOMOG_SHIFT || h->aniso || h->links) return HLBM_ERR_STATE;
    DeviceGuard g(h->device);
    const size_t sb = h->state_bytes();
    const size_t N = h->cells;
    const long nsnap = nsteps > 0 ? (nsteps - 1) / every + 1 : 1;
    const int nseg = every > 2 ? every : 2;  // slot 0/1 double as forward ping-pong buffers
    LaunchCtx c = h->ctx(h->stream);
    Scratch sc(h);
    char *snaps = nullptr, *seg = nullptr;
    float *lam_a = nullptr, *lam_b = nullptr, *gacc = nullptr;
    double *jdev = nullptr, *tmp = nullptr;
    HLBM_CUDA(sc.alloc((void**)&snaps, sb * nsnap));
    HLBM_CUDA(sc.alloc((void**)&seg, sb * nseg));
    HLBM_CUDA(sc.alloc((void**)&lam_a, (size_t)h->q * N * sizeof(float)));
    HLBM_CUDA(sc.alloc((void**)&lam_b, (size_t)h->q * N * sizeof(float)));
    HLBM_CUDA(sc.alloc((void**)&gacc, N * sizeof(float)));
    HLBM_CUDA(sc.alloc((void**)&jdev, sizeof(double)));
    if (h->pattern != HLBM_TWO_LATTICE) HLBM_CUDA(sc.alloc((void**)&tmp, (size_t)h->q * N * sizeof(double)));
    OwnStream own;
    HLBM_CUDA(own.fork(h));
    c.stream = own.s;
    int rc = copy_natural(h, c, snaps, tmp);
    if (rc != HLBM_OK) return rc;

    // forward sweep, keeping f^{k*every}, and in the last segment every state: the reverse sweep
    // starts there, so only the segments before it are recomputed (90 steps kept every 45: 134
    // forward steps instead of 178). The final state goes to slot 0, which no segment uses.
    // Where nothing needs the state in between, two steps go in one launch; the single steps and the
    // reverse steps are chained (180 steps of 128^3 kept every 45: 30.4 -> 28.8 ms for the gradient).
    const long last0 = (nsnap - 1) * every;
    const bool two = step2_applies(c);
    void* a = snaps;
    for (long s = 0, flip = 0; s < nsteps;) {
        const bool pair = two && s + 1 < last0 && (s + 1) % every != 0;
        const long n = s + (pair ? 2 : 1);  // the state that this launch produces
        const bool keep = n % every == 0 && n / every < nsnap;
        const long slot = n == nsteps ? 0 : (n > last0 ? n - last0 : (flip ^= 1));
        void* b = keep ? (void*)(snaps + sb * (n / every)) : (void*)(seg + sb * slot);
        if (pair) HLBM_CUDA(launch_step2(c, a, b, h->varpi));
        else HLBM_CUDA(launch_step(c, MODE_TWO_LATTICE, a, b, h->varpi));
        a = b;
        s = n;
        c.chained = CHAIN_STREAM;
    }
    c.chained = CHAIN_NONE;
    HLBM_CUDA(launch_plane_flux(c, kNatural, a, plane_x, jdev));
    rc = adopt_natural(h, c, a, tmp);
    if (rc != HLBM_OK) return rc;

    // reverse sweep
    HLBM_CUDA(launch_flux_seed(c, lam_a, plane_x));
    HLBM_CUDA(cudaMemsetAsync(gacc, 0, N * sizeof(float), c.stream));
    for (long sg = nsnap - 1; sg >= 0 && nsteps > 0; --sg) {
        const long s0 = sg * every;
        const long s1 = s0 + every < nsteps ? s0 + every : nsteps;
        auto state = [&](long k) -> void* { return k == 0 ? (void*)(snaps + sb * sg) : (void*)(seg + sb * k); };
        for (long k = 0; sg + 1 < nsnap && k + 1 < s1 - s0; ++k)
            HLBM_CUDA(launch_step(c, MODE_TWO_LATTICE, state(k), state(k + 1), h->varpi));
        for (long s = s1 - 1; s >= s0; --s) {
            HLBM_CUDA(launch_adjoint_step(c, state(s - s0), lam_a, lam_b, h->varpi, gacc));
            c.chained = CHAIN_STREAM;
            float* t = lam_a;
            lam_a = lam_b;
            lam_b = t;
        }
    }
    HLBM_CUDA(cudaMemcpyAsync(grad, gacc, N * sizeof(float),
                              on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost, c.stream));
    HLBM_CUDA(cudaMemcpyAsync(J, jdev, sizeof(double), cudaMemcpyDeviceToHost, c.stream));
    HLBM_CUDA(cudaStreamSynchronize(c.stream));
    h->step += nsteps;
    return HLBM_OK;
}

int hlbm_save(hlbm_t* h, const char* path) {
    if (!h || !path) return HLBM_ERR_INVALID_ARG;
    DeviceGuard g(h->device);
    std::vector<char> st(h->state_bytes());
    std::vector<float> vp(h->cells);
    HLBM_CUDA(cudaMemcpyAsync(st.data(), h->state(), st.size(), cudaMemcpyDeviceToHost, h->stream));
    HLBM_CUDA(cudaMemcpyAsync(vp.data(), h->varpi, vp.size() * sizeof(float), cudaMemcpyDeviceToHost, h->stream));
    HLBM_CUDA(cudaStreamSynchronize(h->stream));
    CkptHeader hd;
    std::memset(&hd, 0, sizeof(hd));
    std::memcpy(hd.magic, "HLBMCKP1", 8);
    hd.q = h->q;
    hd.nx = h->nx;
    hd.ny = h->ny;
    hd.nz = h->nz;
    hd.storage = h->storage;
    hd.pattern = h->pattern;
    hd.cur = 0;
    hd.aa_odd = h->aa_odd;
    hd.step = h->step;
    hd.tau = h->tau;
    for (int a = 0; a < 3; ++a) {
        hd.F[a] = h->F[a];
        hd.bc[a] = h->bc[a];
    }
    hd.scale = h->scale;
    hd.pad = h->homog;
    FILE* fp = std::fopen(path, "wb");
    if (!fp) return HLBM_ERR_IO;
    bool ok = std::fwrite(&hd, sizeof(hd), 1, fp) == 1 && std::fwrite(st.data(), 1, st.size(), fp) == st.size() &&
              std::fwrite(vp.data(), sizeof(float), vp.size(), fp) == vp.size();
    ok = (std::fclose(fp) == 0) && ok;
    return ok ? HLBM_OK : HLBM_ERR_IO;
}

int hlbm_load(hlbm_t* h, const char* path) {
    if (!h || !path) return HLBM_ERR_INVALID_ARG;
    DeviceGuard g(h->device);
    FILE* fp = std::fopen(path, "rb");
    if (!fp) return HLBM_ERR_IO;
    CkptHeader hd;
    bool ok = std::fread(&hd, sizeof(hd), 1, fp) == 1 && std::memcmp(hd.magic, "HLBMCKP1", 8) == 0;
    ok = ok && hd.q == h->q && hd.nx == h->nx && hd.ny == h->ny && hd.nz == h->nz && hd.storage == h->storage &&
         hd.pattern == h->pattern;
    std::vector<char> st(ok ? h->state_bytes() : 0);
    std::vector<float> vp(ok ? h->cells : 0);
    ok = ok && std::fread(st.data(), 1, st.size(), fp) == st.size() &&
         std::fread(vp.data(), sizeof(float), vp.size(), fp) == vp.size();
    std::fclose(fp);
    if (!ok) return HLBM_ERR_IO;
    if (!(hd.tau > 0.5)) return HLBM_ERR_IO;
    h->cur = 0;
    h->aa_odd = hd.aa_odd;
    h->step = hd.step;
    h->tau = hd.tau;
    for (int a = 0; a < 3; ++a) {
        h->F[a] = hd.F[a];
        h->bc[a] = hd.bc[a];
    }
    h->scale = hd.scale;
    h->homog = hd.pad == HLBM_HOMOG_DRAG ? HLBM_HOMOG_DRAG : HLBM_HOMOG_SHIFT;
    h->settings_changed();
    HLBM_CUDA(cudaMemcpyAsync(h->buf[0], st.data(), st.size(), cudaMemcpyHostToDevice, h->stream));
    HLBM_CUDA(cudaMemcpyAsync(h->varpi, vp.data(), vp.size() * sizeof(float), cudaMemcpyHostToDevice, h->stream));
    HLBM_CUDA(rest_solids(h));
    HLBM_CUDA(cudaMemsetAsync(h->u_prev, 0, 3 * h->cells * h->arith_bytes(), h->stream));
    HLBM_CUDA(cudaStreamSynchronize(h->stream));
    return HLBM_OK;
}

}  // extern "C"
