// Device and pinned host memory of handles and servers, kept between objects.
//
// Creating a lattice took about 0.4 ms, destroying it 0.3 to 1 ms, and the first
// call that needs scratch mapped it again (1.4 ms for a 48^3 gradient over 90
// steps, whose kernels run 1.6 ms): a design loop or a batch of small solves pays
// that for every object. A handle therefore takes its scratch, and its lattice if
// that is small, from a private stream-ordered pool, and a pool that is given back
// is kept for the next handle, trimmed to kKeepBytes; at most kKeepPools are kept, the
// others are destroyed. Servers share one pool that holds up to kKeepBytes unused (a
// slot's memory was mapped at each admission). Pinned blocks are kept likewise, up to
// kKeepPinned bytes. A failed allocation first returns what is kept. What is kept belongs
// to the context that was current when it was allocated, and serves and is returned in that
// context only; up to kContexts contexts of a device keep something, a further one nothing.
// Streams for the length of a call are kept too: a stream created, used and destroyed for each
// gradient made graphs with branches 4 % slower for the rest of the process (series of 200 samples
// of 64^3 2475 -> 2568 us), with a kept one they are not.
// Measured: gradient of a 48^3 box over 90 steps through torch.autograd, handle included,
// 3.80 -> 2.10 ms; submitting a 96^3 request 1.2 -> 0.34 ms.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstring>
#include <map>
#include <mutex>
#include <new>
#include <set>
#include <type_traits>
#include <vector>

#include "internal.h"

namespace hlbm {

namespace {

constexpr int kMaxDevices = 64, kContexts = 4;
static_assert(sizeof(ContextFact::known) / sizeof(ContextFact::known[0]) == kMaxDevices);
// per context:
constexpr size_t kKeepPools = 2, kKeepBytes = (size_t)512 << 20;  // at most 1.5 GiB stays mapped
constexpr size_t kKeepPinned = (size_t)64 << 20;
constexpr size_t kKeepStreams = 4;
constexpr size_t kSlotBytes = 64, kSlots = 256;  // small pinned results (one page-locked block)

struct Kept {
    unsigned long long context = 0;  // id of the context that all of this belongs to; 0: a free record
    cudaMemPool_t pools[kKeepPools] = {};
    size_t npools = 0;
    cudaStream_t streams[kKeepStreams] = {};
    size_t nstreams = 0;
    cudaMemPool_t shared = nullptr;
    std::multimap<size_t, void*> pinned;  // capacity -> block
    size_t pinned_bytes = 0;
    std::set<void*> held;  // pools, pinned blocks and streams that objects have
    char* slots = nullptr;
    std::vector<int> free_slots;
};
std::mutex& kept_mutex() {
    static std::mutex m;
    static_assert(std::is_trivially_destructible_v<std::mutex>, "usable while the process ends");
    return m;
}

// 0: no context is current.
unsigned long long context_id() {
    using GetId = int (*)(void*, unsigned long long*);
    static const GetId get = [] {
        void* f = nullptr;
        cudaDriverEntryPointQueryResult r;
        if (cudaGetDriverEntryPointByVersion("cuCtxGetId", &f, 12000, cudaEnableDefault, &r) != cudaSuccess) f = nullptr;
        return reinterpret_cast<GetId>(f);
    }();
    unsigned long long id = 0;
    if (get && get(nullptr, &id) == 0) return id;
    if (get && cudaFree(nullptr) == cudaSuccess && get(nullptr, &id) == 0) return id;  // creates the context
    (void)cudaGetLastError();
    return 0;
}

// Runs what may lack host memory for its bookkeeping. False: it did, and the object at hand is
// then not kept (these functions are called from the C ABI, which no exception crosses).
template <class Fn>
bool has_memory(Fn&& fn) {
    try {
        fn();
        return true;
    } catch (const std::bad_alloc&) {
        return false;
    }
}

// All records, under kept_mutex(). Never destroyed (objects may be released while the process
// ends), and a record stays its context's: an object may be released with another one current.
struct Records {
    Kept of[kMaxDevices][kContexts];
    Kept* used[kMaxDevices * kContexts] = {};  // those with a context (walking all of them costs 25 us)
    int nused = 0;
};
Records* records() {  // null: out of host memory
    static Records* all = nullptr;
    if (!all) all = new (std::nothrow) Records();
    return all;
}

// What the current context keeps. Null: nothing can be kept.
Kept* kept() {
    int device = -1;
    if (cudaGetDevice(&device) != cudaSuccess || device < 0 || device >= kMaxDevices) return nullptr;
    const unsigned long long id = context_id();
    Records* const all = id ? records() : nullptr;
    if (!all) return nullptr;
    for (Kept& k : all->of[device]) {
        if (k.context == id) return &k;
        if (k.context) continue;
        if (!has_memory([&] { k.free_slots.reserve(kSlots); })) return nullptr;
        k.context = id;
        all->used[all->nused++] = &k;
        return &k;
    }
    return nullptr;
}

// The record that a pool, pinned block or stream is held under, which it is taken off; null: none.
Kept* holder(void* p) {
    Records* const all = records();
    for (int i = 0; all && i < all->nused; ++i)
        if (all->used[i]->held.erase(p)) return all->used[i];
    return nullptr;
}

// Holds a new pool, pinned block or stream under the current context.
void hold(void* p) {
    holder(p);  // a context that is gone may have had one at this address
    if (Kept* const k = kept()) has_memory([&] { k->held.insert(p); });
}

cudaError_t create_pool(unsigned long long hold, cudaMemPool_t* pool) {
    *pool = nullptr;
    cudaMemPoolProps pr;
    std::memset(&pr, 0, sizeof(pr));
    pr.allocType = cudaMemAllocationTypePinned;
    pr.location.type = cudaMemLocationTypeDevice;
    cudaError_t e = cudaGetDevice(&pr.location.id);
    if (e != cudaSuccess) return e;
    e = cudaMemPoolCreate(pool, &pr);
    if (e == cudaSuccess) {
        e = cudaMemPoolSetAttribute(*pool, cudaMemPoolAttrReleaseThreshold, &hold);
        if (e != cudaSuccess) cudaMemPoolDestroy(*pool);
    }
    if (e != cudaSuccess) *pool = nullptr;
    return e;
}

}  // namespace

// All functions here work in the current context.

bool ContextFact::get(int (*ask)()) {
    int device = -1;
    if (cudaGetDevice(&device) != cudaSuccess) return false;
    const unsigned long long id = context_id();
    const bool remembers = id && device >= 0 && device < kMaxDevices;
    if (remembers) {
        const unsigned long long k = known[device].load(std::memory_order_relaxed);
        if (k >> 1 == id) return k & 1;
    }
    const int yes = ask();
    if (remembers && yes >= 0) known[device].store(id * 2 + yes, std::memory_order_relaxed);
    return yes == 1;
}

void memory_give_back() {
    cudaMemPool_t pools[kKeepPools];
    size_t npools = 0;
    std::multimap<size_t, void*> blocks;
    cudaMemPool_t shared = nullptr;
    {
        std::lock_guard<std::mutex> lk(kept_mutex());
        if (Kept* const k = kept()) {
            std::swap(npools, k->npools);
            std::copy(k->pools, k->pools + npools, pools);
            blocks.swap(k->pinned);
            k->pinned_bytes = 0;
            shared = k->shared;
        }
    }
    for (size_t i = 0; i < npools; ++i) cudaMemPoolDestroy(pools[i]);
    if (shared) cudaMemPoolTrimTo(shared, 0);
    for (auto& b : blocks) cudaFreeHost(b.second);
}

bool pool_keeps(size_t bytes) { return bytes <= kKeepBytes; }

cudaError_t pool_acquire(cudaMemPool_t* pool) {
    {
        std::lock_guard<std::mutex> lk(kept_mutex());
        Kept* const k = kept();
        if (k && k->npools) {
            *pool = k->pools[--k->npools];
            has_memory([&] { k->held.insert(*pool); });
            return cudaSuccess;
        }
    }
    const cudaError_t e = create_pool(~0ull, pool);  // hands nothing back on synchronisation
    if (e != cudaSuccess) return e;
    std::lock_guard<std::mutex> lk(kept_mutex());
    hold(*pool);
    return cudaSuccess;
}

cudaError_t pool_shared(cudaMemPool_t* pool, bool* own) {
    *pool = nullptr;
    *own = false;
    std::lock_guard<std::mutex> lk(kept_mutex());
    Kept* const k = kept();
    if (!k) {  // nothing is kept here
        *own = true;
        return create_pool(kKeepBytes, pool);
    }
    if (!k->shared) {
        const cudaError_t e = create_pool(kKeepBytes, &k->shared);
        if (e != cudaSuccess) return e;
    }
    *pool = k->shared;
    return cudaSuccess;
}

void pool_release(cudaMemPool_t pool) {
    if (!pool) return;
    const bool trimmed = cudaMemPoolTrimTo(pool, kKeepBytes) == cudaSuccess;
    {
        std::lock_guard<std::mutex> lk(kept_mutex());
        Kept* const k = holder(pool);
        if (trimmed && k && k->npools < kKeepPools) {
            k->pools[k->npools++] = pool;
            return;
        }
    }
    cudaMemPoolDestroy(pool);
}

cudaError_t stream_acquire(cudaStream_t* s) {
    {
        std::lock_guard<std::mutex> lk(kept_mutex());
        Kept* const k = kept();
        if (k && k->nstreams) {
            *s = k->streams[--k->nstreams];
            has_memory([&] { k->held.insert(*s); });
            return cudaSuccess;
        }
    }
    const cudaError_t e = cudaStreamCreateWithFlags(s, cudaStreamNonBlocking);
    if (e != cudaSuccess) {
        *s = nullptr;
        return e;
    }
    std::lock_guard<std::mutex> lk(kept_mutex());
    hold(*s);
    return cudaSuccess;
}

void stream_release(cudaStream_t s, bool idle) {
    {
        std::lock_guard<std::mutex> lk(kept_mutex());
        Kept* const k = holder(s);
        if (idle && k && k->nstreams < kKeepStreams) {
            k->streams[k->nstreams++] = s;
            return;
        }
    }
    cudaStreamDestroy(s);
}

cudaError_t pool_alloc(cudaMemPool_t pool, void** p, size_t bytes, cudaStream_t s) {
    cudaError_t e = cudaMallocFromPoolAsync(p, bytes, pool, s);
    if (e == cudaErrorMemoryAllocation) {
        (void)cudaGetLastError();
        memory_give_back();
        e = cudaMallocFromPoolAsync(p, bytes, pool, s);
    }
    return e;
}

cudaError_t device_malloc(void** p, size_t bytes) {
    cudaError_t e = cudaMalloc(p, bytes);
    if (e == cudaErrorMemoryAllocation) {
        (void)cudaGetLastError();
        memory_give_back();
        e = cudaMalloc(p, bytes);
    }
    return e;
}

void* pinned_acquire(size_t bytes, size_t* capacity) {
    {
        std::lock_guard<std::mutex> lk(kept_mutex());
        if (Kept* const k = kept()) {
            const auto it = k->pinned.lower_bound(bytes);
            if (it != k->pinned.end() && it->first <= 2 * bytes) {
                void* b = it->second;
                *capacity = it->first;
                k->pinned_bytes -= it->first;
                k->pinned.erase(it);
                has_memory([&] { k->held.insert(b); });
                return b;
            }
        }
    }
    void* b = nullptr;
    *capacity = bytes;
    cudaError_t e = cudaMallocHost(&b, bytes);
    if (e != cudaSuccess) {
        (void)cudaGetLastError();
        memory_give_back();
        e = cudaMallocHost(&b, bytes);
    }
    if (e != cudaSuccess) {
        (void)cudaGetLastError();
        return nullptr;
    }
    std::lock_guard<std::mutex> lk(kept_mutex());
    hold(b);
    return b;
}

void pinned_release(void* b, size_t capacity) {
    if (!b) return;
    {
        std::lock_guard<std::mutex> lk(kept_mutex());
        Kept* const k = holder(b);
        if (k && k->pinned_bytes + capacity <= kKeepPinned && has_memory([&] { k->pinned.emplace(capacity, b); })) {
            k->pinned_bytes += capacity;
            return;
        }
    }
    cudaFreeHost(b);
}

// 64 bytes of pinned memory.
double* slot_acquire() {
    void* b = nullptr;
    {
        std::lock_guard<std::mutex> lk(kept_mutex());
        Kept* const k = kept();
        if (k && !k->slots && cudaHostAlloc(&b, kSlotBytes * kSlots, cudaHostAllocPortable) == cudaSuccess) {
            k->slots = static_cast<char*>(b);
            for (int i = (int)kSlots - 1; i >= 0; --i) k->free_slots.push_back(i);
        }
        if (k && !k->free_slots.empty()) {
            const int i = k->free_slots.back();
            k->free_slots.pop_back();
            return reinterpret_cast<double*>(k->slots + (size_t)i * kSlotBytes);
        }
    }
    if (cudaMallocHost(&b, kSlotBytes) == cudaSuccess) return static_cast<double*>(b);
    (void)cudaGetLastError();
    return nullptr;
}

void slot_release(double* p) {
    if (!p) return;
    char* const c = reinterpret_cast<char*>(p);
    {
        std::lock_guard<std::mutex> lk(kept_mutex());
        Records* const all = records();
        for (int i = 0; all && i < all->nused; ++i) {
            Kept& k = *all->used[i];
            if (k.slots && c >= k.slots && c < k.slots + kSlotBytes * kSlots) {  // never freed: others use the block
                k.free_slots.push_back((int)((c - k.slots) / kSlotBytes));
                return;
            }
        }
    }
    cudaFreeHost(p);
}

}  // namespace hlbm
