// csrc/api.cu on the CPU: the file is linked with fakes of the CUDA calls and kernel launches that
// it makes, which write down what is launched where and what a graph holds. The argument names the
// case to run; the exit status is 0 when it holds, and a line on stderr says what does not.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <set>
#include <vector>

#include "../../include/hlbm.h"
#include "internal.h"

namespace {

struct Launch {
    const char* kernel;
    cudaStream_t stream;
    int chained;
};
std::vector<Launch> g_log;       // launches, copies and graph launches outside captures, in order
std::set<cudaStream_t> g_capturing;
size_t g_nodes = 0;              // kernels in the graph that is being captured
std::vector<size_t> g_graphs;    // kernels of each graph that was instantiated (an executable graph's handle, too)
size_t g_next = 0;               // handles of the fake objects
int g_failed = 0;

void expect(bool ok, const char* what, long a = 0, long b = 0) {
    if (ok) return;
    if (!g_failed) std::fprintf(stderr, "failed: %s (%ld, %ld)\n", what, a, b);
    g_failed = 1;
}
template <class T>
T fresh() {
    return reinterpret_cast<T>(g_next += 16);
}
cudaError_t record(const char* kernel, cudaStream_t s, int chained = 0) {
    if (g_capturing.count(s)) ++g_nodes;
    else g_log.push_back({kernel, s, chained});
    return cudaSuccess;
}
cudaError_t allocate(void** p, size_t n) {
    *p = std::calloc(1, n);
    return cudaSuccess;
}

}  // namespace

extern "C" {

const char* cudaGetErrorName(cudaError_t) { return "error"; }
const char* cudaGetErrorString(cudaError_t) { return "error"; }
cudaError_t cudaGetLastError(void) { return cudaSuccess; }
cudaError_t cudaGetDevice(int* d) { return *d = 0, cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaFree(void* p) { return std::free(p), cudaSuccess; }
cudaError_t cudaFreeAsync(void* p, cudaStream_t) { return std::free(p), cudaSuccess; }
cudaError_t cudaDeviceSynchronize(void) { return cudaSuccess; }
cudaError_t cudaMemPoolTrimTo(cudaMemPool_t, size_t) { return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { return *s = fresh<cudaStream_t>(), cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t, unsigned) { return record("wait", s); }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return *e = fresh<cudaEvent_t>(), cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus* c) {
    return *c = cudaStreamCaptureStatusNone, cudaSuccess;
}
cudaError_t cudaStreamBeginCapture(cudaStream_t s, cudaStreamCaptureMode) {
    g_nodes = 0;
    return g_capturing.insert(s), cudaSuccess;
}
cudaError_t cudaStreamEndCapture(cudaStream_t s, cudaGraph_t* g) {
    g_capturing.erase(s);
    return *g = fresh<cudaGraph_t>(), cudaSuccess;
}
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* e, cudaGraph_t, unsigned long long) {
    g_graphs.push_back(g_nodes);
    return *e = reinterpret_cast<cudaGraphExec_t>(g_nodes), cudaSuccess;
}
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t e, cudaStream_t s) {
    return record(reinterpret_cast<size_t>(e) == 8 ? "graph 8" : "graph 16", s);
}
cudaError_t cudaMemcpyAsync(void*, const void*, size_t, cudaMemcpyKind, cudaStream_t s) { return record("copy", s); }
cudaError_t cudaMemsetAsync(void*, int, size_t, cudaStream_t s) { return record("set", s); }

}  // extern "C"

namespace hlbm {

bool pool_keeps(size_t) { return true; }
cudaError_t pool_acquire(cudaMemPool_t* p) { return *p = fresh<cudaMemPool_t>(), cudaSuccess; }
void pool_release(cudaMemPool_t) {}
cudaError_t stream_acquire(cudaStream_t* s) { return cudaStreamCreateWithFlags(s, 0); }
void stream_release(cudaStream_t, bool) {}
cudaError_t pool_alloc(cudaMemPool_t, void** p, size_t n, cudaStream_t) { return allocate(p, n); }
cudaError_t device_malloc(void** p, size_t n) { return allocate(p, n); }
double* slot_acquire() { return static_cast<double*>(std::malloc(64)); }
void slot_release(double* p) { std::free(p); }
void memory_give_back() {}
size_t storage_bytes(int storage) { return storage == 0 ? 8 : (storage == 1 ? 4 : 2); }
size_t reduce_partials_count(const LaunchCtx&) { return 8; }
bool step2_applies(const LaunchCtx&) { return false; }
bool resident_applies(const LaunchCtx&) { return false; }

cudaError_t launch_step(const LaunchCtx& c, int, const void*, void*, const float*) { return record("step", c.stream, c.chained); }
cudaError_t launch_step2(const LaunchCtx& c, const void*, void*, const float*) { return record("step2", c.stream); }
cudaError_t launch_resident(const LaunchCtx& c, void*, const float*, int) { return record("resident", c.stream); }
cudaError_t launch_adjoint_step(const LaunchCtx& c, const void*, const float*, float*, const float*, float*) {
    return record("reverse step", c.stream, c.chained);
}
cudaError_t launch_flux_seed(const LaunchCtx& c, float*, int) { return record("seed", c.stream); }
cudaError_t launch_plane_flux(const LaunchCtx& c, int, const void*, int, double*) { return record("flux", c.stream); }
cudaError_t launch_reduce(const LaunchCtx& c, int, const void*, void*, int, double*, double*) { return record("reduce", c.stream); }
cudaError_t launch_moments(const LaunchCtx& c, int, const void*, void*, void*, int) { return record("moments", c.stream); }
cudaError_t launch_build_links(const LaunchCtx& c, const unsigned char*, unsigned*) { return record("links", c.stream); }
cudaError_t launch_rest_solid(const LaunchCtx& c, void*) { return record("rest", c.stream); }
cudaError_t launch_write_state(const LaunchCtx& c, int, const double*, int, void*) { return record("write", c.stream); }
cudaError_t launch_read_state(const LaunchCtx& c, int, const void*, double*) { return record("read", c.stream); }
cudaError_t launch_check_unit_interval(const float*, size_t, int*, cudaStream_t s) { return record("check", s); }
cudaError_t launch_fill_f32(float*, size_t, float, cudaStream_t s) { return record("fill", s); }

}  // namespace hlbm

namespace {

hlbm_t* lattice(int pattern, cudaStream_t stream) {
    hlbm_t* h = nullptr;
    expect(hlbm_create(&h, 19, 24, 24, 24, HLBM_F32, pattern, stream) == HLBM_OK, "create");
    return h;
}
long count(const char* kernel) {
    return std::count_if(g_log.begin(), g_log.end(), [&](const Launch& l) { return !std::strcmp(l.kernel, kernel); });
}

// A run after a change of a setting captures no more than the short graph, until the present
// settings have been used for long; then the long graph serves, and every step is taken.
void captures() {
    hlbm_t* h = lattice(HLBM_TWO_LATTICE, fresh<cudaStream_t>());
    for (const long n : {7, 8, 15, 16, 24, 31, 32, 48, 80}) {
        expect(hlbm_set_force(h, 1e-5 * n, 0, 0) == HLBM_OK, "set_force");
        g_graphs.clear();
        g_log.clear();
        expect(hlbm_step(h, n) == HLBM_OK, "step");
        size_t nodes = 0;
        for (const size_t g : g_graphs) nodes += g;
        expect(nodes <= 8, "kernels captured for a run after a change", n, (long)nodes);
        expect(8 * count("graph 8") + 16 * count("graph 16") + count("step") == n, "steps", n);
        if (n % 2) hlbm_step(h, 1);
    }
    for (const long n : {16, 24, 100, 128, 200, 1000}) {
        hlbm_set_force(h, 2e-5 * n, 0, 0);
        for (int k = 0; k < 100; ++k) {
            g_log.clear();
            g_graphs.clear();
            hlbm_step(h, n);
            expect(8 * count("graph 8") + 16 * count("graph 16") + count("step") == n, "steps of a repeated run", n, k);
        }
        expect(g_graphs.empty(), "nothing is captured again", n);
        expect(count("graph 16") == n / 16 && count("graph 8") == n % 16 / 8, "the fewest replays", n);
    }
    hlbm_destroy(h);
}

// The chained kernels of a gradient follow one another on a stream that is not the caller's, and the
// first of a row follows the work that comes before it plainly.
void gradient() {
    cudaStream_t const stream = fresh<cudaStream_t>();
    for (const int pattern : {HLBM_TWO_LATTICE, HLBM_AA}) {
        hlbm_t* h = lattice(pattern, stream);
        std::vector<float> grad(24 * 24 * 24);
        double J = 0.0;
        g_log.clear();
        expect(hlbm_adjoint_flux_grad(h, 11, 4, 12, &J, grad.data(), 0) == HLBM_OK, "gradient");
        long steps = 0;
        for (size_t k = 0; k < g_log.size(); ++k) {
            const Launch& l = g_log[k];
            const bool sweep = !std::strcmp(l.kernel, "step") || !std::strcmp(l.kernel, "reverse step");
            steps += sweep;
            expect(!sweep || l.stream != stream, "a sweep off the caller's stream", (long)k);
            if (!l.chained) continue;
            const Launch& before = g_log[k - 1];
            expect(before.stream == l.stream && (!std::strcmp(before.kernel, "step") || !std::strcmp(before.kernel, "reverse step")),
                   "a chained kernel directly follows a kernel", (long)k);
        }
        expect(steps == 11 + 6 + 11, "steps of the sweeps", steps);
        hlbm_destroy(h);
    }
}

}  // namespace

int main(int argc, char** argv) {
    const char* const name = argc > 1 ? argv[1] : "";
    if (!std::strcmp(name, "captures")) captures();
    else if (!std::strcmp(name, "gradient")) gradient();
    else expect(false, "a case of this program");
    return g_failed;
}
