// fake_cudart.cpp -- a CUDA runtime without a device, for the host side of the
// library (test_host_runtime.py links it with the library's objects).  Kernels
// do nothing but are counted by name; memory is the host's, zero, and never
// written by memsets.  What it keeps account of:
//  * stream-ordered allocations: one is ready once its stream, an event behind
//    it or the device has been waited for; a memset or copy that touches it
//    from another stream before that is a violation;
//  * bytes mapped: cudaMalloc's, and what the memory pools hold (freed blocks
//    stay until a wait, above the release threshold, or cudaMemPoolTrimTo), the
//    highest value since the last reset, and a capacity past which allocations
//    fail; the n-th allocation from now on, and some after it, can be made to fail;
//  * waits, graph launches, and whether a stream is capturing.
#include <cuda_runtime.h>
#include <sys/mman.h>

#include <algorithm>
#include <cstring>
#include <map>
#include <mutex>
#include <set>
#include <string>

namespace {

struct Alloc {
    size_t bytes = 0;
    int pool = 0;  // 0: cudaMalloc
    cudaStream_t stream = nullptr;
    bool ready = true;
};
struct Pool {
    size_t used = 0, reserved = 0, keep = 0;
};

std::recursive_mutex mu;
std::map<char *, Alloc> allocs;
std::map<int, Pool> pools;
std::map<const void *, std::string> names;
std::map<std::string, long> launches;
std::set<cudaStream_t> capturing;
size_t malloced = 0, capacity = (size_t)200 << 30, peak = 0;
long violations = 0, fail_after = -1, fail_count = 0, next_id = 1, waits = 0;
dim3 cfg_grid, cfg_block;
size_t cfg_smem;
cudaStream_t cfg_stream;
thread_local cudaError_t last = cudaSuccess;

size_t mapped() {
    size_t n = malloced;
    for (auto &p : pools) n += p.second.reserved;
    return n;
}

cudaError_t fail(cudaError_t e) {
    last = e;
    return e;
}

// Whether an allocation that maps `more` bytes succeeds.
bool room(size_t more) {
    if (fail_after > 0) --fail_after;
    else if (fail_after == 0 && fail_count > 0) { --fail_count; return false; }
    if (mapped() + more > capacity) return false;
    return true;
}

void *host(size_t n) {
    void *p = mmap(nullptr, std::max<size_t>(n, 4096), PROT_READ | PROT_WRITE,
                   MAP_PRIVATE | MAP_ANONYMOUS | MAP_NORESERVE, -1, 0);
    return p == MAP_FAILED ? nullptr : p;
}

void touch(const void *p, cudaStream_t s) {
    auto it = allocs.upper_bound((char *)p);
    if (it == allocs.begin()) return;
    --it;
    if ((char *)p >= it->first + it->second.bytes) return;
    if (!it->second.ready && it->second.stream != s) ++violations;
}

void waited(cudaStream_t s, bool all) {
    ++waits;
    for (auto &a : allocs)
        if (all || a.second.stream == s) a.second.ready = true;
    for (auto &p : pools)
        if (p.second.reserved > std::max(p.second.keep, p.second.used))
            p.second.reserved = std::max(p.second.keep, p.second.used);
}

}  // namespace

#define LOCK std::lock_guard<std::recursive_mutex> lk(mu)

extern "C" {

// ---- what a test asks
long fake_violations() { LOCK; return violations; }
long fake_launches(const char *part) {
    LOCK;
    long n = 0;
    for (auto &l : launches)
        if (l.first.find(part) != std::string::npos) n += l.second;
    return n;
}
long fake_waits() { LOCK; return waits; }
unsigned long long fake_mapped() { LOCK; return mapped(); }
unsigned long long fake_peak() { LOCK; return peak; }
void fake_set_capacity(unsigned long long b) { LOCK; capacity = b; }
void fake_fail_after(long n, long count) { LOCK; fail_after = n; fail_count = count; }
void fake_capture(void *s, int on) { LOCK; if (on) capturing.insert((cudaStream_t)s); else capturing.erase((cudaStream_t)s); }
void fake_reset() {
    LOCK;
    launches.clear();
    violations = 0;
    peak = mapped();
    fail_after = -1;
    waits = 0;
}

// ---- registration and launches
void **__cudaRegisterFatBinary(void *) { static void *h; return &h; }
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterFunction(void **, const char *f, char *, const char *name, int, uint3 *, uint3 *,
                            dim3 *, dim3 *, int *) {
    LOCK;
    names[f] = name;
}
void __cudaRegisterVar(void **, char *, char *, const char *, int, size_t, int, int) {}
cudaError_t __cudaGetKernel(cudaKernel_t *k, const void *f) { *k = (cudaKernel_t)f; return cudaSuccess; }
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t sm, CUstream_st *s) {
    cfg_grid = g; cfg_block = b; cfg_smem = sm; cfg_stream = s;
    return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3 *g, dim3 *b, size_t *sm, void *s) {
    *g = cfg_grid; *b = cfg_block; *sm = cfg_smem; *(cudaStream_t *)s = cfg_stream;
    return cudaSuccess;
}
cudaError_t cudaLaunchKernel(const void *f, dim3, dim3, void **, size_t, cudaStream_t) {
    LOCK;
    ++launches[names[f]];
    return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 g, dim3 b, void **a, size_t sm, cudaStream_t s) {
    return cudaLaunchKernel((const void *)k, g, b, a, sm, s);
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *, const void *f, void **) {
    LOCK;
    ++launches[names[f]];
    return cudaSuccess;
}

// ---- device
cudaError_t cudaGetDeviceCount(int *n) { *n = 1; return cudaSuccess; }
cudaError_t cudaGetDevice(int *d) { *d = 0; return cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr, int) { *v = 152; return cudaSuccess; }
cudaError_t cudaGetDeviceProperties(cudaDeviceProp *p, int) {
    std::memset(p, 0, sizeof(*p));
    p->multiProcessorCount = 152;
    return cudaSuccess;
}
cudaError_t cudaDeviceSynchronize() { LOCK; waited(nullptr, true); return cudaSuccess; }
cudaError_t cudaMemGetInfo(size_t *f, size_t *t) { LOCK; *t = capacity; *f = capacity - mapped(); return cudaSuccess; }
cudaError_t cudaGetLastError() { cudaError_t e = last; last = cudaSuccess; return e; }
cudaError_t cudaPeekAtLastError() { return last; }
const char *cudaGetErrorString(cudaError_t) { return "fake"; }
cudaError_t cudaFuncSetAttribute(const void *, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessor(int *n, const void *, int, size_t) { *n = 3; return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int *n, const void *, int, size_t, unsigned) { *n = 3; return cudaSuccess; }
cudaError_t cudaGetSymbolAddress(void **, const void *) { return fail(cudaErrorInvalidSymbol); }

// ---- memory
cudaError_t cudaMalloc(void **p, size_t n) {
    LOCK;
    if (!room(n)) return fail(cudaErrorMemoryAllocation);
    *p = host(n);
    allocs[(char *)*p] = Alloc{n, 0, nullptr, true};
    malloced += n;
    peak = std::max(peak, mapped());
    return cudaSuccess;
}
cudaError_t cudaFree(void *p) {
    LOCK;
    waited(nullptr, true);
    auto it = allocs.find((char *)p);
    if (it == allocs.end()) return fail(cudaErrorInvalidValue);
    if (it->second.pool) pools[it->second.pool].used -= it->second.bytes; else malloced -= it->second.bytes;
    munmap(p, std::max<size_t>(it->second.bytes, 4096));
    allocs.erase(it);
    return cudaSuccess;
}
cudaError_t cudaHostAlloc(void **p, size_t n, unsigned) { *p = host(n); return cudaSuccess; }
cudaError_t cudaFreeHost(void *) { return cudaSuccess; }
cudaError_t cudaMemPoolCreate(cudaMemPool_t *p, const cudaMemPoolProps *) {
    LOCK;
    *p = (cudaMemPool_t)next_id;
    pools[(int)next_id++];
    return cudaSuccess;
}
cudaError_t cudaMemPoolDestroy(cudaMemPool_t p) { LOCK; pools.erase((int)(long)p); return cudaSuccess; }
cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t p, cudaMemPoolAttr a, void *v) {
    LOCK;
    if (a == cudaMemPoolAttrReleaseThreshold) pools[(int)(long)p].keep = *(unsigned long long *)v;
    return cudaSuccess;
}
cudaError_t cudaMemPoolGetAttribute(cudaMemPool_t p, cudaMemPoolAttr a, void *v) {
    LOCK;
    Pool &q = pools[(int)(long)p];
    if (a == cudaMemPoolAttrUsedMemCurrent) *(unsigned long long *)v = q.used;
    if (a == cudaMemPoolAttrReservedMemCurrent) *(unsigned long long *)v = q.reserved;
    return cudaSuccess;
}
cudaError_t cudaMemPoolTrimTo(cudaMemPool_t p, size_t keep) {
    LOCK;
    Pool &q = pools[(int)(long)p];
    q.reserved = std::min(q.reserved, std::max(q.used, keep));
    return cudaSuccess;
}
cudaError_t cudaMallocFromPoolAsync(void **p, size_t n, cudaMemPool_t pool, cudaStream_t s) {
    LOCK;
    Pool &q = pools[(int)(long)pool];
    const size_t more = q.used + n > q.reserved ? q.used + n - q.reserved : 0;
    if (!room(more)) return fail(cudaErrorMemoryAllocation);
    q.used += n;
    q.reserved += more;
    *p = host(n);
    allocs[(char *)*p] = Alloc{n, (int)(long)pool, s, false};
    peak = std::max(peak, mapped());
    return cudaSuccess;
}
cudaError_t cudaFreeAsync(void *p, cudaStream_t) {
    LOCK;
    auto it = allocs.find((char *)p);
    if (it == allocs.end()) return fail(cudaErrorInvalidValue);
    if (it->second.pool) pools[it->second.pool].used -= it->second.bytes; else malloced -= it->second.bytes;
    munmap(p, std::max<size_t>(it->second.bytes, 4096));
    allocs.erase(it);
    return cudaSuccess;
}
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, cudaMemcpyKind) {
    LOCK;
    touch(d, nullptr);
    touch(s, nullptr);
    std::memcpy(d, s, n);
    return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind, cudaStream_t st) {
    LOCK;
    touch(d, st);
    touch(s, st);
    std::memcpy(d, s, n);
    return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void *d, int, size_t, cudaStream_t st) { LOCK; touch(d, st); return cudaSuccess; }

// ---- streams, events, graphs
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) { LOCK; *s = (cudaStream_t)next_id++; return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t s) { LOCK; waited(s, false); return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t s, cudaStreamCaptureMode) { LOCK; capturing.insert(s); return cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t s, cudaGraph_t *g) { LOCK; capturing.erase(s); *g = (cudaGraph_t)next_id++; return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t s, cudaStreamCaptureStatus *st) {
    LOCK;
    *st = capturing.count(s) ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
    return cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t *e, cudaGraph_t, unsigned long long) { LOCK; *e = (cudaGraphExec_t)next_id++; return cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { LOCK; ++launches["graph"]; return cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t *e) { LOCK; *e = (cudaEvent_t)next_id++; return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) { LOCK; *e = (cudaEvent_t)next_id++; return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventRecordWithFlags(cudaEvent_t, cudaStream_t, unsigned) { return cudaSuccess; }
cudaError_t cudaEventQuery(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t, cudaEvent_t) { *ms = 1.0f; return cudaSuccess; }

}  // extern "C"
