// Device memory of the library: one CUDA memory pool per device, shared by every handle
// and every call. Allocation is stream-ordered and thread-safe (the driver's), and the
// pool keeps up to POOL_KEEP freed bytes mapped: mapping and unmapping a call's working
// states (8 GiB at 24 qubits) took 19 ms of each call, and the five buffers of an error
// list 0.2 ms with cudaMalloc. When the last circuit or surrogate handle is freed, all but
// POOL_IDLE goes back: a program that makes one handle at a time would otherwise map its
// memory anew for each (0.7 ms of a surrogate's 2.8).
//
// Two pools a device. Working memory is freed on the stream (or the idle stream) that
// allocated it, and only that one reuses it: with the driver's search among the blocks of
// other streams on, an allocation grew by 50 us over some thirty streams (surrogate
// 1.9 -> 3.7 ms in a long process). A block that another stream holds back goes home when
// the pool exceeds POOL_KEEP, or when an allocation fails for want of it. Error lists
// outlive their stream: made on it, freed on the idle one, they keep that search.
#include <atomic>
#include <mutex>

#include "internal.h"

namespace arso {

constexpr uint64_t POOL_KEEP = 17ull << 30;  // the largest working set of one call (16 GiB) and the handles' tables
constexpr uint64_t POOL_IDLE = 256ull << 20;
constexpr uint64_t LIST_KEEP = 1ull << 30, LIST_IDLE = 64ull << 20;
constexpr int MAX_DEVICES = 64;

namespace {
struct DevicePool {
    std::mutex mu;
    cudaMemPool_t pool = nullptr, lists = nullptr;
    cudaStream_t idle = nullptr;  // never runs anything: frees and allocations on it complete at once
};
DevicePool g_pools[MAX_DEVICES];
std::atomic<long> g_handles{0};

DevicePool &device_pool() {
    int dev = 0;
    ARSO_CUDA(cudaGetDevice(&dev));
    ARSO_REQUIRE(dev >= 0 && dev < MAX_DEVICES, "device index out of range");
    DevicePool &p = g_pools[dev];
    std::lock_guard<std::mutex> lk(p.mu);
    if (!p.pool) {
        cudaMemPoolProps props{};
        props.allocType = cudaMemAllocationTypePinned;
        props.location.type = cudaMemLocationTypeDevice;
        props.location.id = dev;
        uint64_t keep = POOL_KEEP, keep_lists = LIST_KEEP;
        int off = 0;
        if (!p.idle) ARSO_CUDA(cudaStreamCreateWithFlags(&p.idle, cudaStreamNonBlocking));
        if (!p.lists) ARSO_CUDA(cudaMemPoolCreate(&p.lists, &props));
        ARSO_CUDA(cudaMemPoolSetAttribute(p.lists, cudaMemPoolAttrReleaseThreshold, &keep_lists));
        cudaMemPool_t pool = nullptr;
        ARSO_CUDA(cudaMemPoolCreate(&pool, &props));
        p.pool = pool;
        ARSO_CUDA(cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep));
        ARSO_CUDA(cudaMemPoolSetAttribute(pool, cudaMemPoolReuseAllowOpportunistic, &off));
        ARSO_CUDA(cudaMemPoolSetAttribute(pool, cudaMemPoolReuseAllowInternalDependencies, &off));
    }
    return p;
}

void *alloc_from(cudaMemPool_t pool, DevicePool &p, size_t bytes, cudaStream_t st) {
    void *ptr = nullptr;
    cudaError_t e = cudaMallocFromPoolAsync(&ptr, bytes, pool, st);
    if (e == cudaErrorMemoryAllocation) {  // what other streams hold back goes home first
        cudaGetLastError();
        cudaDeviceSynchronize();
        cudaMemPoolTrimTo(p.pool, 0);
        cudaMemPoolTrimTo(p.lists, 0);
        e = cudaMallocFromPoolAsync(&ptr, bytes, pool, st);
    }
    ARSO_CUDA(e);
    return ptr;
}
}  // namespace

void *pool_alloc(size_t bytes, cudaStream_t st) {
    DevicePool &p = device_pool();
    return alloc_from(p.pool, p, bytes, st);
}

void *pool_alloc_list(size_t bytes, cudaStream_t st) {
    DevicePool &p = device_pool();
    return alloc_from(p.lists, p, bytes, st);
}

void *pool_alloc_now(size_t bytes) {
    DevicePool &p = device_pool();
    void *ptr = alloc_from(p.pool, p, bytes, p.idle);
    const cudaError_t e = cudaStreamSynchronize(p.idle);
    if (e != cudaSuccess) {
        cudaFreeAsync(ptr, p.idle);
        ARSO_CUDA(e);
    }
    return ptr;
}

void pool_free_idle(void *ptr) noexcept {
    if (!ptr) return;
    try {
        cudaFreeAsync(ptr, device_pool().idle);
    } catch (...) {
        cudaFree(ptr);
    }
}

void handle_made() { g_handles.fetch_add(1); }
void handle_freed() noexcept {
    if (g_handles.fetch_sub(1) != 1) return;
    for (DevicePool &p : g_pools) {
        std::lock_guard<std::mutex> lk(p.mu);
        if (!p.pool) continue;
        cudaStreamSynchronize(p.idle);
        cudaMemPoolTrimTo(p.pool, POOL_IDLE);
        cudaMemPoolTrimTo(p.lists, LIST_IDLE);
    }
}

}  // namespace arso
