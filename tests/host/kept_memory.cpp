// csrc/mem.cu on the CPU: the file is linked with the fake CUDA calls below, which know the
// current context, what is allocated and what is freed. The argument names the case to run;
// the exit status is 0 when it holds, and a line on stderr says what does not.
#include <cuda_runtime.h>

#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <new>
#include <set>

#include "internal.h"

namespace {

unsigned long long g_context = 1;  // id of the current context
bool g_have_ids = true;            // does the driver know context ids?
std::map<char*, size_t> g_pinned;  // page-locked blocks that are allocated
std::set<cudaMemPool_t> g_pools;   // pools that exist
size_t g_next_pool = 16;
int g_failed = 0;
bool g_no_memory = false;  // operator new fails

int fake_ctx_get_id(void*, unsigned long long* id) {
    *id = g_context;
    return g_context ? 0 : 201;
}
void expect(bool ok, const char* what) {
    if (ok) return;
    std::fprintf(stderr, "failed: %s\n", what);
    g_failed = 1;
}
// Is [p, p + n) page-locked?
bool mapped(const void* p, size_t n) {
    const char* c = static_cast<const char*>(p);
    for (const auto& b : g_pinned)
        if (c >= b.first && c + n <= b.first + b.second) return true;
    return false;
}
cudaError_t host_alloc(void** p, size_t n) {
    const bool no_memory = g_no_memory;
    g_no_memory = false;  // for the list below
    *p = std::malloc(n);
    g_pinned[static_cast<char*>(*p)] = n;
    g_no_memory = no_memory;
    return cudaSuccess;
}

}  // namespace

void* operator new(size_t n) {
    if (g_no_memory) throw std::bad_alloc();
    return std::malloc(n ? n : 1);
}
void* operator new(size_t n, const std::nothrow_t&) noexcept { return g_no_memory ? nullptr : std::malloc(n ? n : 1); }
void operator delete(void* p) noexcept { std::free(p); }
void operator delete(void* p, size_t) noexcept { std::free(p); }

extern "C" {

cudaError_t cudaGetDevice(int* d) {
    *d = 0;
    return cudaSuccess;
}
cudaError_t cudaGetLastError(void) { return cudaSuccess; }
cudaError_t cudaGetDriverEntryPointByVersion(const char*, void** f, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult* r) {
    *f = g_have_ids ? reinterpret_cast<void*>(&fake_ctx_get_id) : nullptr;
    *r = g_have_ids ? cudaDriverEntryPointSuccess : cudaDriverEntryPointSymbolNotFound;
    return g_have_ids ? cudaSuccess : cudaErrorSymbolNotFound;
}
cudaError_t cudaFree(void*) { return cudaSuccess; }
cudaError_t cudaMalloc(void** p, size_t n) {
    *p = std::malloc(n);
    return cudaSuccess;
}
cudaError_t cudaMallocHost(void** p, size_t n) { return host_alloc(p, n); }
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned) { return host_alloc(p, n); }
cudaError_t cudaFreeHost(void* p) {
    const auto it = g_pinned.find(static_cast<char*>(p));
    expect(it != g_pinned.end(), "only the start of an allocated page-locked block is freed");
    if (it == g_pinned.end()) return cudaErrorInvalidValue;
    std::free(p);
    g_pinned.erase(it);
    return cudaSuccess;
}
cudaError_t cudaMemPoolCreate(cudaMemPool_t* p, const cudaMemPoolProps*) {
    const bool no_memory = g_no_memory;
    g_no_memory = false;
    *p = reinterpret_cast<cudaMemPool_t>(g_next_pool += 16);
    g_pools.insert(*p);
    g_no_memory = no_memory;
    return cudaSuccess;
}
cudaError_t cudaMemPoolDestroy(cudaMemPool_t p) {
    expect(g_pools.erase(p) == 1, "only an existing pool is destroyed");
    return cudaSuccess;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) {
    *s = reinterpret_cast<cudaStream_t>(g_next_pool += 16);
    return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t, cudaMemPoolAttr, void*) { return cudaSuccess; }
cudaError_t cudaMemPoolTrimTo(cudaMemPool_t p, size_t) {
    expect(g_pools.count(p) == 1, "only an existing pool is trimmed");
    return cudaSuccess;
}
cudaError_t cudaMallocFromPoolAsync(void** p, size_t n, cudaMemPool_t, cudaStream_t) {
    *p = std::malloc(n);
    return cudaSuccess;
}

}  // extern "C"

namespace {

using namespace hlbm;

// A driver without context ids: nothing can be kept, and everything still works.
void no_context_ids() {
    g_have_ids = false;
    cudaMemPool_t a = nullptr, b = nullptr;
    expect(pool_acquire(&a) == cudaSuccess && a, "a handle gets a pool");
    bool own = false;
    expect(pool_shared(&b, &own) == cudaSuccess && b && b != a && own, "a server gets a pool of its own");
    if (own) cudaMemPoolDestroy(b);
    pool_release(a);
    size_t capacity = 0;
    void* p = pinned_acquire(1000, &capacity);
    expect(p && mapped(p, 1000), "a page-locked block");
    pinned_release(p, capacity);
    double* s = slot_acquire();
    expect(s && mapped(s, 64), "a slot");
    slot_release(s);
    expect(g_pinned.empty() && g_pools.empty(), "everything is returned");
}

// Objects of several contexts on one device, released in any order and with any context current.
void several_contexts() {
    double* const a = slot_acquire();
    double* const b = slot_acquire();
    cudaMemPool_t pool = nullptr, other = nullptr, again = nullptr;
    pool_acquire(&pool);
    pool_release(pool);
    size_t ca = 0, cb = 0;
    void* const pa = pinned_acquire(1000, &ca);
    void* const pb = pinned_acquire(1000, &cb);
    pinned_release(pa, ca);

    g_context = 2;
    double* const c = slot_acquire();
    expect(c && c != a && c != b, "a slot of its own in the second context");
    pool_acquire(&other);
    expect(other != pool, "a pool of its own in the second context");
    void* const pc = pinned_acquire(1000, &ca);
    expect(pc != pa, "a page-locked block of its own in the second context");
    pinned_release(pb, cb);  // of the first context

    g_context = 1;
    slot_release(a);
    expect(mapped(b, 64) && mapped(c, 64), "the other handles keep their slots");
    *b = 1.0;
    pool_acquire(&again);
    expect(again == pool, "the pool of the first context serves again");
    pool_release(other);  // of the second context
    expect(pool_acquire(&other) == cudaSuccess && g_pools.size() == 3, "and no pool of another one");
    pool_release(other);
    pool_release(again);
    slot_release(c);
    slot_release(b);
    pinned_release(pc, ca);
    expect(slot_acquire() == b && slot_acquire() == a, "released slots serve again");
    void* const p1 = pinned_acquire(1000, &ca);
    void* const p2 = pinned_acquire(1000, &cb);
    expect((p1 == pa && p2 == pb) || (p1 == pb && p2 == pa), "blocks go back to the context that they come from");

    cudaStream_t s1 = nullptr, s2 = nullptr, s3 = nullptr;
    stream_acquire(&s1);
    stream_acquire(&s2);
    expect(s1 && s2 && s1 != s2, "a stream for each call");
    stream_release(s2, false);
    g_context = 2;
    stream_release(s1, true);
    stream_acquire(&s3);
    expect(s3 != s1 && s3 != s2, "a stream of the second context");
    g_context = 1;
    stream_acquire(&s2);
    expect(s1 == s2, "an idle stream of the first context serves again");
    stream_release(s2, true);
    stream_release(s3, true);

    for (g_context = 3; g_context < 10; ++g_context) {  // more contexts than are kept for
        cudaMemPool_t p = nullptr;
        double* const s = slot_acquire();
        expect(pool_acquire(&p) == cudaSuccess && p && s && mapped(s, 64), "a handle in any context");
        pool_release(p);
        slot_release(s);
    }
    expect(g_pools.size() <= 2 * 4, "a bounded number of pools stays");
}

// Host memory runs out at any call: nothing is thrown, and what cannot be kept is freed.
void no_host_memory() {
    for (int fail_from = 0; fail_from < 4; ++fail_from) {
        g_no_memory = fail_from == 0;
        cudaMemPool_t p = nullptr;
        size_t capacity = 0;
        bool own = false;
        cudaMemPool_t shared = nullptr;
        expect(pool_shared(&shared, &own) == cudaSuccess, "a server gets a pool");
        if (own) cudaMemPoolDestroy(shared);
        g_no_memory = fail_from <= 1;
        expect(pool_acquire(&p) == cudaSuccess, "a handle gets a pool");
        void* const b = pinned_acquire(1000, &capacity);
        double* const s = slot_acquire();
        expect(b && mapped(b, 1000) && s && mapped(s, 64), "and page-locked memory");
        g_no_memory = fail_from <= 2;
        pool_release(p);
        pinned_release(b, capacity);
        slot_release(s);
        memory_give_back();
    }
    g_no_memory = false;
    expect(g_pools.size() == 1 && g_pinned.size() == 1, "the servers' pool and the slots stay, nothing else");
}

// A fact is asked once per context, of the context that is current, and an error is not remembered.
int g_asked = 0, g_answer = 1;
void context_facts() {
    static ContextFact fact;
    const auto ask = [] { return ++g_asked, g_answer; };
    expect(fact.get(ask) && fact.get(ask) && g_asked == 1, "asked once");
    g_context = 2;
    g_answer = 0;
    expect(!fact.get(ask) && !fact.get(ask) && g_asked == 2, "another context is asked, and has its own answer");
    g_context = 1;
    g_answer = 1;
    expect(fact.get(ask), "the first context keeps its answer");
    g_context = 3;
    g_answer = -1;
    expect(!fact.get(ask), "an error is a no");
    g_answer = 1;
    expect(fact.get(ask), "that is not remembered");
    g_context = 0;
    g_answer = 0;
    expect(!fact.get(ask), "no context");
}

}  // namespace

int main(int argc, char** argv) {
    const char* const name = argc > 1 ? argv[1] : "";
    if (!std::strcmp(name, "no_context_ids")) no_context_ids();
    else if (!std::strcmp(name, "several_contexts")) several_contexts();
    else if (!std::strcmp(name, "no_host_memory")) no_host_memory();
    else if (!std::strcmp(name, "context_facts")) context_facts();
    else expect(false, "a case of this program");
    return g_failed;
}
