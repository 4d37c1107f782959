// A CUDA runtime for tests of the library's host code on a machine without a GPU:
// "device" memory is host memory with an unmapped range after every allocation,
// copies and memsets are checked against the allocations they touch, kernel
// launches are recorded by name and do nothing, and a test may watch or fail any
// call (fake_hook). Linked with the library's own objects in place of the CUDA
// runtime (tests/host_library.py).
#include <cuda_runtime.h>
#include <sys/mman.h>

#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <mutex>
#include <string>

// (device intrinsics that common.cuh names; nothing here calls them)
double __longlong_as_double(long long);
long long __double_as_longlong(double);
#include "common.cuh"

namespace {

constexpr size_t GUARD = size_t(1) << 24;  // unmapped bytes after an allocation
struct Alloc {
    bool data;
    size_t bytes, mapped;  // mapped: from the allocation's start to the end of its guard
};
std::recursive_mutex mu;
std::map<uintptr_t, Alloc> allocs;
std::string faults;
// (by call: kernels register while the library's other objects are still being set up)
std::string &kernel(const void *fn) {
    static std::map<const void *, std::string> names;
    return names[fn];
}
cudaError_t last = cudaSuccess;
typedef int (*Hook)(const char *call, const char *what, uint64_t bytes);
Hook hook = nullptr;

// The hook sees every call; a nonzero answer is the call's error.
cudaError_t ask(const char *call, const char *what = "", uint64_t bytes = 0) {
    const int e = hook ? hook(call, what, bytes) : 0;
    if (e) last = (cudaError_t)e;
    return (cudaError_t)e;
}

uintptr_t up(size_t n) { return (n + 4095) / 4096 * 4096; }

// Allocations end at a page's end when `bytes` is a multiple of 256, so that
// overruns are caught by the range checks and, by the host, as a fault.
cudaError_t get(void **p, size_t bytes) {
    std::lock_guard<std::recursive_mutex> lk(mu);
    const size_t room = up(bytes), mapped = room + GUARD;
    void *m = mmap(nullptr, mapped, PROT_NONE, MAP_PRIVATE | MAP_ANONYMOUS | MAP_NORESERVE, -1, 0);
    if (m == MAP_FAILED || mprotect(m, room, PROT_READ | PROT_WRITE)) return last = cudaErrorMemoryAllocation;
    const uintptr_t at = (uintptr_t)m + (room - bytes) / 256 * 256;
    allocs[at] = Alloc{false, bytes, (uintptr_t)m + mapped - at};
    *p = (void *)at;
    return cudaSuccess;
}

// 0: not device memory; 1: [p, p + n) lies in one allocation; 2: it runs past one.
int where(const void *p, size_t n) {
    std::lock_guard<std::recursive_mutex> lk(mu);
    auto it = allocs.upper_bound((uintptr_t)p);
    if (it == allocs.begin()) return 0;
    --it;
    const uintptr_t off = (uintptr_t)p - it->first;
    if (off >= it->second.mapped) return 0;
    return off + n <= it->second.bytes ? 1 : 2;
}
bool inside(const char *call, const void *p, size_t n) {
    if (where(p, n) != 2) return true;
    std::lock_guard<std::recursive_mutex> lk(mu);
    auto it = --allocs.upper_bound((uintptr_t)p);
    char line[160];
    snprintf(line, sizeof line, "%s: %zu bytes at offset %zu of an allocation of %zu\n", call, n,
             (size_t)((uintptr_t)p - it->first), it->second.bytes);
    faults += line;
    return false;
}
cudaError_t copy(void *d, const void *s, size_t n) {
    if (cudaError_t e = ask("cudaMemcpy", "", n)) return e;
    if (inside("copy to", d, n) && inside("copy from", s, n) && n) memmove(d, s, n);
    return cudaSuccess;
}
cudaError_t fill(void *d, int v, size_t n) {
    if (inside("memset", d, n) && n) memset(d, v, n);
    return cudaSuccess;
}
cudaError_t launch(const void *fn) {
    std::string name;
    {
        std::lock_guard<std::recursive_mutex> lk(mu);
        name = kernel(fn);
    }
    return ask("launch", name.c_str());
}

}  // namespace

extern "C" {

// ---- for the tests ------------------------------------------------------------------
void fake_hook(Hook h) { hook = h; }
int fake_where(const void *p, size_t n) { return where(p, n); }
const char *fake_faults() { return faults.c_str(); }
void fake_clear_faults() { faults.clear(); }
// The device allocation of `bytes` bytes (the lowest if several); null if none.
void *fake_find(size_t bytes) {
    for (auto &a : allocs)
        if (a.second.bytes == bytes) return (void *)a.first;
    return nullptr;
}
// The allocation at p holds a test's own data (two column indices can look like a pointer).
void fake_data(void *p) {
    std::lock_guard<std::recursive_mutex> lk(mu);
    allocs.at((uintptr_t)p).data = true;
}
// Words of the library's device memory that point past the end of an allocation.
int fake_stray_pointers() {
    std::lock_guard<std::recursive_mutex> lk(mu);
    int n = 0;
    for (auto &a : allocs)
        for (size_t k = 0; k + 8 <= a.second.bytes && !a.second.data; k += 8) {
            const void *p;
            memcpy(&p, (const char *)a.first + k, 8);
            n += where(p, 1) == 2;
        }
    return n;
}
size_t fake_state_bytes() { return sizeof(rbs::SolverState); }
size_t fake_state_done() { return offsetof(rbs::SolverState, done); }
size_t fake_state_iter() { return offsetof(rbs::SolverState, iter); }

// ---- memory -------------------------------------------------------------------------
cudaError_t cudaMalloc(void **p, size_t n) {
    if (cudaError_t e = ask("cudaMalloc", "", n)) return e;
    return get(p, n);
}
cudaError_t cudaFree(void *p) {
    std::lock_guard<std::recursive_mutex> lk(mu);
    auto it = allocs.find((uintptr_t)p);
    if (it != allocs.end()) {  // the range stays reserved: a stale pointer never meets a new allocation
        const uintptr_t page = it->first / 4096 * 4096, end = it->first + it->second.mapped;
        mmap((void *)page, end - page, PROT_NONE, MAP_FIXED | MAP_PRIVATE | MAP_ANONYMOUS | MAP_NORESERVE, -1, 0);
        allocs.erase(it);
    }
    return cudaSuccess;
}
cudaError_t cudaMallocAsync(void **p, size_t n, cudaStream_t) { return cudaMalloc(p, n); }
cudaError_t cudaMallocFromPoolAsync(void **p, size_t n, cudaMemPool_t, cudaStream_t) { return cudaMalloc(p, n); }
cudaError_t cudaFreeAsync(void *p, cudaStream_t) { return cudaFree(p); }
cudaError_t cudaMallocHost(void **p, size_t n) { return (*p = calloc(1, n ? n : 1)) ? cudaSuccess : cudaErrorMemoryAllocation; }
cudaError_t cudaHostAlloc(void **p, size_t n, unsigned) { return cudaMallocHost(p, n); }
cudaError_t cudaFreeHost(void *p) { free(p); return cudaSuccess; }
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, cudaMemcpyKind) { return copy(d, s, n); }
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind, cudaStream_t) { return copy(d, s, n); }
cudaError_t cudaMemcpy2DAsync(void *d, size_t dp, const void *s, size_t sp, size_t w, size_t h, cudaMemcpyKind, cudaStream_t) {
    for (size_t i = 0; i < h; i++) copy((char *)d + i * dp, (const char *)s + i * sp, w);
    return cudaSuccess;
}
cudaError_t cudaMemset(void *d, int v, size_t n) { return fill(d, v, n); }
cudaError_t cudaMemsetAsync(void *d, int v, size_t n, cudaStream_t) { return fill(d, v, n); }
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes *a, const void *p) {
    memset(a, 0, sizeof *a);
    a->type = where(p, 1) ? cudaMemoryTypeDevice : cudaMemoryTypeUnregistered;
    return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void **p, const void *) { return get(p, 8192); }
cudaError_t cudaMemPoolCreate(cudaMemPool_t *p, const cudaMemPoolProps *) { *p = (cudaMemPool_t)1; return cudaSuccess; }
cudaError_t cudaMemPoolDestroy(cudaMemPool_t) { return cudaSuccess; }
cudaError_t cudaMemPoolGetAttribute(cudaMemPool_t, cudaMemPoolAttr, void *v) { *(int64_t *)v = 0; return cudaSuccess; }
cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t, cudaMemPoolAttr, void *) { return cudaSuccess; }

// ---- device, streams, events, graphs -------------------------------------------------
cudaError_t cudaGetDevice(int *d) { *d = 0; return cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaDeviceSynchronize() { return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr a, int) {
    *v = a == cudaDevAttrMultiProcessorCount ? 152 : a == cudaDevAttrMaxSharedMemoryPerBlockOptin ? 232448 : 0;
    return cudaSuccess;
}
cudaError_t cudaGetLastError() { const cudaError_t e = last; last = cudaSuccess; return e; }
const char *cudaGetErrorString(cudaError_t e) { static thread_local char t[32]; snprintf(t, sizeof t, "fake error %d", (int)e); return t; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) { static uintptr_t n = 16; *s = (cudaStream_t)(n += 16); return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return ask("cudaStreamSynchronize"); }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaSuccess; }
cudaError_t cudaStreamBeginCaptureToGraph(cudaStream_t, cudaGraph_t, const cudaGraphNode_t *, const cudaGraphEdgeData *, size_t, cudaStreamCaptureMode) { return cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t *g) { *g = (cudaGraph_t)1; return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t *e) { *e = (cudaEvent_t)1; return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventQuery(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t, cudaEvent_t) { *ms = 1.f; return cudaSuccess; }
cudaError_t cudaGraphCreate(cudaGraph_t *g, unsigned) { *g = (cudaGraph_t)1; return cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaGraphConditionalHandleCreate(cudaGraphConditionalHandle *h, cudaGraph_t, unsigned, unsigned) { *h = 1; return cudaSuccess; }
cudaError_t cudaGraphAddNode(cudaGraphNode_t *n, cudaGraph_t, const cudaGraphNode_t *, const cudaGraphEdgeData *, size_t, cudaGraphNodeParams *p) {
    static cudaGraph_t body[1] = {(cudaGraph_t)2};
    *n = (cudaGraphNode_t)1;
    p->conditional.phGraph_out = body;
    return cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t *x, cudaGraph_t, unsigned long long) { *x = (cudaGraphExec_t)1; return cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return ask("cudaGraphLaunch"); }

// ---- kernels ------------------------------------------------------------------------
cudaError_t cudaFuncGetAttributes(cudaFuncAttributes *a, const void *) { memset(a, 0, sizeof *a); return cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void *fn, cudaFuncAttribute a, int v) {
    return ask(a == cudaFuncAttributePreferredSharedMemoryCarveout ? "carveout" : "cudaFuncSetAttribute", kernel(fn).c_str(), (uint64_t)(int64_t)v);
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int *n, const void *, int, size_t, unsigned) { *n = 3; return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveClusters(int *n, const void *, const cudaLaunchConfig_t *) { *n = 8; return cudaSuccess; }
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *, const void *fn, void **) { return launch(fn); }
cudaError_t __cudaGetKernel(cudaKernel_t *k, const void *fn) { *k = (cudaKernel_t)fn; return cudaSuccess; }
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3, dim3, void **, size_t, cudaStream_t) { return launch((const void *)k); }
unsigned __cudaPushCallConfiguration(dim3, dim3, size_t, cudaStream_t) { return 0; }
cudaError_t __cudaPopCallConfiguration(dim3 *, dim3 *, size_t *, void *) { return cudaSuccess; }
void **__cudaRegisterFatBinary(void *) { static void *h; return &h; }
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
char __cudaInitModule(void **) { return 1; }
void __cudaRegisterVar(void **, char *, char *, const char *, int, size_t, int, int) {}
void __cudaRegisterFunction(void **, const char *host, char *, const char *name, int, uint3 *, uint3 *, dim3 *, dim3 *, int *) {
    std::lock_guard<std::recursive_mutex> lk(mu);
    kernel(host) = name;
}

}  // extern "C"
