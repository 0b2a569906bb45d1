// Device memory of the library: one CUDA memory pool per context (the device's primary one,
// unless a caller makes others), shared by every handle and every call. Allocation is
// stream-ordered and thread-safe (the driver's), and the pool keeps up to POOL_KEEP freed
// bytes mapped: mapping and unmapping a call's working states (8 GiB at 24 qubits) took
// 19 ms of each call, and the five buffers of an error list 0.2 ms with cudaMalloc. When the
// last circuit or surrogate handle is freed, all but POOL_IDLE goes back: a program that makes
// one handle at a time would otherwise map its memory anew for each (0.7 ms of a surrogate's
// 2.8).
//
// Two pools a context. Working memory is freed on the stream (or the idle stream) that
// allocated it, and only that one reuses it: with the driver's search among the blocks of
// other streams on, an allocation grew by 50 us over some thirty streams (surrogate
// 1.9 -> 3.7 ms in a long process). A block that another stream holds back goes home when
// the pool exceeds POOL_KEEP, or when an allocation fails for want of it. Error lists
// outlive their stream: made on it, freed on the idle one, they keep that search.
//
// A block remembers the pools it came from: it is freed in their context, whichever device or
// context is current then, and not at all when that context is gone (its memory went with it).
// Contexts are told apart by the driver's identifier, which is never used twice, so a device
// reset leaves no pool behind that a later call would take.
#include <atomic>
#include <mutex>

#include <cuda.h>

#include "internal.h"

namespace arso {

constexpr uint64_t POOL_KEEP = 17ull << 30;  // the largest working set of one call (16 GiB) and the handles' tables
constexpr uint64_t POOL_IDLE = 256ull << 20;
constexpr uint64_t LIST_KEEP = 1ull << 30, LIST_IDLE = 64ull << 20;

struct ContextPools {
    CUcontext ctx = nullptr;
    unsigned long long id = 0;
    cudaMemPool_t pool = nullptr, lists = nullptr;
    cudaStream_t idle = nullptr;  // never runs anything: frees and allocations on it complete at once
};

namespace {
std::atomic<long> g_handles{0};
std::mutex g_mu;  // of the list below; its entries stay as they are once made
std::vector<std::unique_ptr<ContextPools>> &all_pools() {
    static auto *v = new std::vector<std::unique_ptr<ContextPools>>();  // handles may outlive static objects
    return *v;
}

struct Driver {
    CUresult (*get_current)(CUcontext *) = nullptr;
    CUresult (*get_id)(CUcontext, unsigned long long *) = nullptr;
    CUresult (*push)(CUcontext) = nullptr;
    CUresult (*pop)(CUcontext *) = nullptr;
};
void entry(const char *name, unsigned version, void **fn) {
    cudaDriverEntryPointQueryResult q{};
    ARSO_CUDA(cudaGetDriverEntryPointByVersion(name, fn, version, cudaEnableDefault, &q));
    if (q != cudaDriverEntryPointSuccess || !*fn) throw Error(ARSO_ECUDA, std::string(name) + " is unavailable");
}
const Driver &driver() {
    static const Driver d = [] {
        Driver x;
        entry("cuCtxGetCurrent", 4000, reinterpret_cast<void **>(&x.get_current));
        entry("cuCtxGetId", 12000, reinterpret_cast<void **>(&x.get_id));
        entry("cuCtxPushCurrent", 4000, reinterpret_cast<void **>(&x.push));
        entry("cuCtxPopCurrent", 4000, reinterpret_cast<void **>(&x.pop));
        return x;
    }();
    return d;
}

// The current context and its identifier; a thread that has none yet gets its device's.
unsigned long long current_id(CUcontext &c) {
    const Driver &d = driver();
    unsigned long long id = 0;
    if (d.get_current(&c) != CUDA_SUCCESS || !c) {
        ARSO_CUDA(cudaFree(nullptr));
        if (d.get_current(&c) != CUDA_SUCCESS) throw Error(ARSO_ECUDA, "no current context");
    }
    if (d.get_id(c, &id) != CUDA_SUCCESS) throw Error(ARSO_ECUDA, "cuCtxGetId failed");
    return id;
}

// The owner's context made current, unless it is or is gone.
struct In {
    bool alive = false, pushed = false;
    explicit In(const ContextPools *p) noexcept {
        try {
            const Driver &d = driver();
            CUcontext c = nullptr;
            unsigned long long id = 0;
            if (d.get_current(&c) == CUDA_SUCCESS && c && d.get_id(c, &id) == CUDA_SUCCESS && id == p->id) {
                alive = true;
            } else if (d.get_id(p->ctx, &id) == CUDA_SUCCESS && id == p->id) {
                alive = pushed = d.push(p->ctx) == CUDA_SUCCESS;
            }
        } catch (...) {
        }
    }
    ~In() {
        CUcontext c;
        if (pushed) driver().pop(&c);
    }
};

ContextPools *context_pools() {
    CUcontext ctx = nullptr;
    const unsigned long long id = current_id(ctx);
    std::lock_guard<std::mutex> lk(g_mu);
    for (auto &p : all_pools())
        if (p->id == id) return p.get();
    std::unique_ptr<ContextPools> p(new ContextPools());
    p->ctx = ctx;
    p->id = id;
    cudaMemPoolProps props{};
    props.allocType = cudaMemAllocationTypePinned;
    props.location.type = cudaMemLocationTypeDevice;
    ARSO_CUDA(cudaGetDevice(&props.location.id));
    uint64_t keep = POOL_KEEP, keep_lists = LIST_KEEP;
    int off = 0;
    ARSO_CUDA(cudaStreamCreateWithFlags(&p->idle, cudaStreamNonBlocking));
    ARSO_CUDA(cudaMemPoolCreate(&p->lists, &props));
    ARSO_CUDA(cudaMemPoolSetAttribute(p->lists, cudaMemPoolAttrReleaseThreshold, &keep_lists));
    ARSO_CUDA(cudaMemPoolCreate(&p->pool, &props));
    ARSO_CUDA(cudaMemPoolSetAttribute(p->pool, cudaMemPoolAttrReleaseThreshold, &keep));
    ARSO_CUDA(cudaMemPoolSetAttribute(p->pool, cudaMemPoolReuseAllowOpportunistic, &off));
    ARSO_CUDA(cudaMemPoolSetAttribute(p->pool, cudaMemPoolReuseAllowInternalDependencies, &off));
    all_pools().push_back(std::move(p));
    return all_pools().back().get();
}

void *alloc_from(cudaMemPool_t pool, const ContextPools *p, size_t bytes, cudaStream_t st) {
    void *ptr = nullptr;
    cudaError_t e = cudaMallocFromPoolAsync(&ptr, bytes, pool, st);
    if (e == cudaErrorMemoryAllocation) {  // what other streams hold back goes home first
        cudaGetLastError();
        cudaDeviceSynchronize();
        cudaMemPoolTrimTo(p->pool, 0);
        cudaMemPoolTrimTo(p->lists, 0);
        e = cudaMallocFromPoolAsync(&ptr, bytes, pool, st);
    }
    ARSO_CUDA(e);
    return ptr;
}
}  // namespace

void *pool_alloc(size_t bytes, cudaStream_t st) {
    const ContextPools *p = context_pools();
    return alloc_from(p->pool, p, bytes, st);
}

void *pool_alloc_list(size_t bytes, cudaStream_t st, ContextPools *&owner) {
    owner = context_pools();
    return alloc_from(owner->lists, owner, bytes, st);
}

void *pool_alloc_now(size_t bytes, ContextPools *&owner) {
    owner = context_pools();
    void *ptr = alloc_from(owner->pool, owner, bytes, owner->idle);
    const cudaError_t e = cudaStreamSynchronize(owner->idle);
    if (e != cudaSuccess) {
        cudaFreeAsync(ptr, owner->idle);
        ARSO_CUDA(e);
    }
    return ptr;
}

void pool_free(void *ptr, ContextPools *owner, bool wait) noexcept {
    In in(owner);
    if (!in.alive) return;
    if (wait) cudaDeviceSynchronize();
    cudaFreeAsync(ptr, owner->idle);
}

unsigned long long context_id() {
    CUcontext c = nullptr;
    return current_id(c);
}

void handle_made() { g_handles.fetch_add(1); }
void handle_freed() noexcept {
    if (g_handles.fetch_sub(1) != 1) return;
    std::lock_guard<std::mutex> lk(g_mu);
    for (auto &p : all_pools()) {
        In in(p.get());
        if (!in.alive) continue;
        cudaStreamSynchronize(p->idle);
        cudaMemPoolTrimTo(p->pool, POOL_IDLE);
        cudaMemPoolTrimTo(p->lists, LIST_IDLE);
    }
}

}  // namespace arso
