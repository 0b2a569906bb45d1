// A CUDA runtime without a GPU, for tests of the library's host side: linked with the library's
// own objects in place of the real runtime. Memory is host memory (zeroed), copies are made at
// once, kernels do nothing. It keeps account of what the real one would do later, and of what
// may not happen then:
//   fake_violation(0)  a kernel on another stream launched while a pageable copy or memset on the
//                      legacy stream may be under way
//   fake_violation(1)  memory freed on a stream while work of another stream of its device is pending
//   fake_violation(2)  memory freed while a device other than its own is current, on another
//                      device's stream, or with a runtime call that waits for another device
//   fake_violation(3)  a use of a pool or stream of a context that is gone
//   fake_violation(4)  a launch with more than 48 KiB of dynamic shared memory in a context where
//                      that was not allowed to the kernel
#include <cuda.h>
#include <cuda_runtime.h>
#include <sys/mman.h>

#include <cstdint>
#include <cstdlib>
#include <cstring>
#include <map>
#include <mutex>
#include <set>
#include <string>
#include <vector>

namespace {
struct Ctx { int dev; uint64_t id; };
struct Stream { Ctx *ctx; uint64_t ctx_id; };
struct Pool { Ctx *ctx; uint64_t ctx_id; };
struct Block { size_t bytes; Ctx *ctx; uint64_t ctx_id; };
std::recursive_mutex mu;
uint64_t next_id = 1;
Ctx ctxs[2] = {{0, 1}, {1, 2}};
int cur = 0;                             // current device
std::set<void *> pending[2];             // streams with work not waited for (legacy: nullptr)
bool legacy_copy[2] = {false, false};
std::map<void *, Block> blocks;
uint64_t violations[5], trims, frees, largest;
long fail_at = -1, allocs = 0;           // the pool allocation that fails (and its retry)
long fail_launch = -1, launches = 0;     // the launch that fails
bool retry_fails = false;
std::vector<std::string> launched;
std::map<const void *, std::string> names;
std::map<std::pair<const void *, uint64_t>, int> allowed;  // dynamic shared memory of (kernel, context)
cudaError_t last = cudaSuccess;

cudaError_t err(cudaError_t e) { if (e != cudaSuccess) last = e; return e; }
void *key(cudaStream_t s) { return s == cudaStreamLegacy ? nullptr : (void *)s; }
int dev_of(cudaStream_t s) {
    if (!key(s) || s == cudaStreamPerThread) return cur;
    Stream *x = reinterpret_cast<Stream *>(s);
    if (x->ctx->id != x->ctx_id) ++violations[3];
    return x->ctx->dev;
}
void work(cudaStream_t s) { pending[dev_of(s)].insert(key(s)); }
void *take(size_t n, Ctx *c) {
    void *p = mmap(nullptr, n ? n : 1, PROT_READ | PROT_WRITE, MAP_PRIVATE | MAP_ANONYMOUS | MAP_NORESERVE, -1, 0);
    blocks[p] = {n, c, c->id};
    if (n > largest) largest = n;
    return p;
}
void drop(void *p) {
    auto it = blocks.find(p);
    if (it == blocks.end()) return;
    munmap(p, it->second.bytes ? it->second.bytes : 1);
    blocks.erase(it);
    ++frees;
}
const Block *block_of(const void *p) {
    auto it = blocks.upper_bound(const_cast<void *>(p));
    if (it == blocks.begin()) return nullptr;
    --it;
    return (const char *)p < (const char *)it->first + it->second.bytes ? &it->second : nullptr;
}
cudaError_t launch(const void *f, size_t smem, cudaStream_t s) {
    std::lock_guard<std::recursive_mutex> g(mu);
    const int d = dev_of(s);
    if (launches++ == fail_launch) return err(cudaErrorLaunchOutOfResources);
    if (legacy_copy[d] && key(s)) ++violations[0];
    if (smem > 48 * 1024 && (size_t)allowed[{f, ctxs[d].id}] < smem) ++violations[4];
    launched.push_back(names.count(f) ? names[f] : "?");
    work(s);
    return cudaSuccess;
}
thread_local struct { dim3 g, b; size_t sm; cudaStream_t s; } call;
}  // namespace

extern "C" {
// ------------------------------------------------------------- the test's side --
uint64_t fake_violation(int k) { return violations[k]; }
uint64_t fake_trims() { return trims; }
uint64_t fake_frees() { return frees; }
uint64_t fake_largest() { return largest; }
uint64_t fake_live() { return blocks.size(); }
uint64_t fake_allocs() { return (uint64_t)allocs; }
uint64_t fake_launches(const char *part) {
    uint64_t n = 0;
    for (const std::string &s : launched) n += s.find(part) != std::string::npos;
    return n;
}
void fake_reset_counts() { memset(violations, 0, sizeof violations), trims = frees = largest = 0, allocs = 0, launched.clear(); }
void fake_fail_at(long k) { fail_at = k, allocs = 0, retry_fails = false; }
void fake_fail_launch_at(long k) { fail_launch = k, launches = 0; }
uint64_t fake_tried() { return (uint64_t)launches; }
void fake_device(int d) { cur = d; }
int fake_current() { return cur; }
void *fake_stream(int d) { return new Stream{&ctxs[d], ctxs[d].id}; }
void fake_device_reset(int d) { ctxs[d].id = 100 + next_id++; pending[d].clear(); legacy_copy[d] = false; }

// ------------------------------------------------------------------ driver ----
static CUresult ctx_current(CUcontext *c) { *c = reinterpret_cast<CUcontext>(&ctxs[cur]); return CUDA_SUCCESS; }
static CUresult ctx_id(CUcontext c, unsigned long long *id) { *id = (c ? reinterpret_cast<Ctx *>(c) : &ctxs[cur])->id; return CUDA_SUCCESS; }
static std::vector<int> below;  // devices under the current one
static CUresult ctx_push(CUcontext c) { below.push_back(cur), cur = reinterpret_cast<Ctx *>(c)->dev; return CUDA_SUCCESS; }
static CUresult ctx_pop(CUcontext *c) { *c = reinterpret_cast<CUcontext>(&ctxs[cur]), cur = below.back(), below.pop_back(); return CUDA_SUCCESS; }
static CUresult encode(...) { return CUDA_SUCCESS; }
cudaError_t cudaGetDriverEntryPointByVersion(const char *name, void **fn, unsigned int, unsigned long long,
                                             cudaDriverEntryPointQueryResult *q) {
    const std::string n = name;
    *fn = n == "cuCtxGetCurrent" ? (void *)ctx_current : n == "cuCtxGetId" ? (void *)ctx_id
        : n == "cuCtxPushCurrent" ? (void *)ctx_push : n == "cuCtxPopCurrent" ? (void *)ctx_pop
        : n == "cuTensorMapEncodeTiled" ? (void *)encode : nullptr;
    if (q) *q = *fn ? cudaDriverEntryPointSuccess : cudaDriverEntryPointSymbolNotFound;
    return cudaSuccess;
}

// ------------------------------------------------------------------ runtime ----
void **__cudaRegisterFatBinary(void *) { static void *h; return &h; }
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterFunction(void **, const char *host, char *, const char *name, int, uint3 *, uint3 *, dim3 *, dim3 *, int *) { names[host] = name; }
void __cudaRegisterVar(void **, char *, char *, const char *, int, size_t, int, int) {}
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t sm, cudaStream_t s) { call = {g, b, sm, s}; return 0; }
cudaError_t __cudaPopCallConfiguration(dim3 *g, dim3 *b, size_t *sm, void *s) {
    *g = call.g, *b = call.b, *sm = call.sm, *(cudaStream_t *)s = call.s;
    return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t *k, const void *f) { *k = (cudaKernel_t)f; return cudaSuccess; }
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3, dim3, void **, size_t sm, cudaStream_t s) { return launch((const void *)k, sm, s); }
cudaError_t cudaLaunchKernel(const void *f, dim3, dim3, void **, size_t sm, cudaStream_t s) { return launch(f, sm, s); }

cudaError_t cudaGetDevice(int *d) { *d = cur; return cudaSuccess; }
cudaError_t cudaSetDevice(int d) { cur = d; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr, int) { *v = 152; return cudaSuccess; }
cudaError_t cudaDeviceSynchronize() { pending[cur].clear(), legacy_copy[cur] = false; return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t s) {
    std::lock_guard<std::recursive_mutex> g(mu);
    const int d = dev_of(s);
    pending[d].erase(key(s));
    if (!key(s)) legacy_copy[d] = false;
    return cudaSuccess;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) { *s = (cudaStream_t)fake_stream(cur); return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return err(cudaErrorStreamCaptureUnsupported); }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t *) { return err(cudaErrorStreamCaptureUnsupported); }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t *, cudaGraph_t, unsigned long long) { return cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t *e) { *e = (cudaEvent_t)0x10; return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t, cudaEvent_t) { *ms = 1.f; return cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void *f, cudaFuncAttribute, int v) { allowed[{f, ctxs[cur].id}] = v; return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessor(int *n, const void *, int, size_t) { *n = 2; return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int *n, const void *, int, size_t, unsigned) { *n = 2; return cudaSuccess; }
cudaError_t cudaGetLastError() { const cudaError_t e = last; last = cudaSuccess; return e; }
const char *cudaGetErrorString(cudaError_t) { return "fake error"; }
cudaError_t cudaGetSymbolAddress(void **p, const void *s) { *p = const_cast<void *>(s); return cudaSuccess; }
cudaError_t cudaMemcpyFromSymbol(void *d, const void *, size_t n, size_t, cudaMemcpyKind) { memset(d, 0, n); return cudaSuccess; }
cudaError_t cudaMemcpyToSymbol(const void *, const void *, size_t, size_t, cudaMemcpyKind) { return cudaSuccess; }
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes *a, const void *p) {
    memset(a, 0, sizeof *a);
    a->type = block_of(p) ? cudaMemoryTypeDevice : cudaMemoryTypeUnregistered;
    return cudaSuccess;
}
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, cudaMemcpyKind k) {
    std::lock_guard<std::recursive_mutex> g(mu);
    memcpy(d, s, n);
    if (k == cudaMemcpyHostToDevice) legacy_copy[cur] = true;
    else pending[cur].erase(nullptr), legacy_copy[cur] = false;
    return cudaSuccess;
}
cudaError_t cudaMemset(void *d, int v, size_t n) {
    std::lock_guard<std::recursive_mutex> g(mu);
    memset(d, v, n);
    legacy_copy[cur] = true;
    return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind, cudaStream_t st) {
    std::lock_guard<std::recursive_mutex> g(mu);
    if (n < (64u << 20)) memcpy(d, s, n);
    work(st);
    return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void *d, int v, size_t n, cudaStream_t st) {
    std::lock_guard<std::recursive_mutex> g(mu);
    if (n < (64u << 20)) memset(d, v, n);
    work(st);
    return cudaSuccess;
}
cudaError_t cudaMemPoolCreate(cudaMemPool_t *p, const cudaMemPoolProps *) { *p = (cudaMemPool_t) new Pool{&ctxs[cur], ctxs[cur].id}; return cudaSuccess; }
cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t, cudaMemPoolAttr, void *) { return cudaSuccess; }
cudaError_t cudaMemPoolTrimTo(cudaMemPool_t, size_t) { ++trims; return cudaSuccess; }
cudaError_t cudaMallocFromPoolAsync(void **p, size_t n, cudaMemPool_t pool, cudaStream_t st) {
    std::lock_guard<std::recursive_mutex> g(mu);
    Pool *q = (Pool *)pool;
    if (q->ctx->id != q->ctx_id) ++violations[3];
    (void)dev_of(st);
    if (retry_fails || allocs++ == fail_at) {
        retry_fails = !retry_fails;  // the call after it is the retry
        return err(cudaErrorMemoryAllocation);
    }
    *p = take(n, q->ctx);
    return cudaSuccess;
}
cudaError_t cudaFreeAsync(void *p, cudaStream_t st) {
    std::lock_guard<std::recursive_mutex> g(mu);
    const auto it = blocks.find(p);
    if (it == blocks.end()) return cudaSuccess;
    const int d = it->second.ctx->dev;
    if (it->second.ctx->id != it->second.ctx_id) ++violations[3];
    if (dev_of(st) != d || cur != d) ++violations[2];
    for (void *x : pending[d])
        if (x != key(st)) {
            ++violations[1];
            break;
        }
    drop(p);
    return cudaSuccess;
}
cudaError_t cudaFree(void *p) {
    std::lock_guard<std::recursive_mutex> g(mu);
    if (p) cudaDeviceSynchronize(), drop(p);
    return cudaSuccess;
}
}  // extern "C"
