// A host-memory stand-in for the CUDA calls that creating and destroying a plan makes, so that what they do with
// device memory is tested without a device: two contexts, an out-of-memory limit, work in flight, captures.
// Linked with the library's host sources; launches do nothing.
#include <cstdint>
#include <cstdlib>
#include <cstring>
#include <map>
#include <new>
#include <string>

#include <cuda.h>
#include <cuda_runtime.h>

#include "launch.h"

namespace {

struct Block {
    size_t bytes;
    unsigned long long context;
};
std::map<void *, Block> g_live;
size_t g_live_bytes, g_limit;
long g_calls_left = -1, g_mallocs, g_frees, g_foreign_frees, g_foreign_writes, g_writes_while_busy;
unsigned long long g_primary, g_current;      // context ids; the primary one is current unless another was pushed
unsigned long long g_next_id = 1;
bool g_busy, g_forbid_malloc, g_capture_elsewhere, g_capture_broken;
cudaError_t g_last;

// counts down the calls that make something; the one that reaches zero fails
bool fails() { return g_calls_left > 0 && --g_calls_left == 0; }
cudaError_t ret(cudaError_t e) { return e == cudaSuccess ? e : (g_last = e); }

CUresult get_id(CUcontext c, unsigned long long *id) { return *id = c ? reinterpret_cast<unsigned long long>(c) : g_current, CUDA_SUCCESS; }
CUresult get_state(CUdevice, unsigned *flags, int *active) { return *flags = 0, *active = 1, CUDA_SUCCESS; }
CUresult retain(CUcontext *c, CUdevice) { return *c = reinterpret_cast<CUcontext>(g_primary), CUDA_SUCCESS; }
CUresult release(CUdevice) { return CUDA_SUCCESS; }
CUresult get_device(CUdevice *d, int i) { return *d = i, CUDA_SUCCESS; }

size_t g_host_limit = SIZE_MAX;

}  // namespace

// of the library's sources alone (hidden): one allocation of more than the limit fails
void *operator new(size_t n) {
    void *p = n > g_host_limit ? nullptr : malloc(n);
    if (!p) throw std::bad_alloc();
    return p;
}
void *operator new(size_t n, const std::nothrow_t &) noexcept { return n > g_host_limit ? nullptr : malloc(n); }
void operator delete(void *p) noexcept { free(p); }
void operator delete(void *p, size_t) noexcept { free(p); }

extern "C" {

// ---- the test's side
__attribute__((visibility("default"))) void fake_fail_call(long k) { g_calls_left = k; }
__attribute__((visibility("default"))) void fake_host_limit(size_t limit) { g_host_limit = limit; }
__attribute__((visibility("default"))) void fake_reset(size_t limit) {
    for (auto &b : g_live) free(b.first);
    g_live.clear();
    g_live_bytes = 0;
    g_limit = limit;
    g_mallocs = g_frees = g_foreign_frees = g_foreign_writes = g_writes_while_busy = 0;
    g_busy = g_forbid_malloc = g_capture_elsewhere = g_capture_broken = false;
    g_last = cudaSuccess;
    g_primary = g_current = g_next_id++;
}
__attribute__((visibility("default"))) void fake_limit(size_t limit) { g_limit = limit; }
__attribute__((visibility("default"))) void fake_push_other_context() { g_current = g_next_id++; }
__attribute__((visibility("default"))) void fake_pop_context() { g_current = g_primary; }
// cudaDeviceReset: the primary context's memory is gone, the next one has a new id
__attribute__((visibility("default"))) void fake_device_reset() {
    for (auto it = g_live.begin(); it != g_live.end();)
        if (it->second.context == g_primary) {
            g_live_bytes -= it->second.bytes;
            free(it->first);
            it = g_live.erase(it);
        } else {
            ++it;
        }
    g_primary = g_current = g_next_id++;
}
__attribute__((visibility("default"))) void fake_busy(int on) { g_busy = on != 0; }
// a capture that forbids allocation calls on every thread
__attribute__((visibility("default"))) void fake_forbid_malloc(int on) { g_forbid_malloc = on != 0; }
// a thread-local or relaxed capture on another thread: allocation calls are allowed, waiting for the device is not
__attribute__((visibility("default"))) void fake_capture_elsewhere(int on) { g_capture_elsewhere = on != 0; }
__attribute__((visibility("default"))) long fake_count(const char *what) {
    const std::string w = what;
    if (w == "live") return (long)g_live.size();
    if (w == "live_bytes") return (long)g_live_bytes;
    if (w == "mallocs") return g_mallocs;
    if (w == "frees") return g_frees;
    if (w == "foreign_frees") return g_foreign_frees;
    if (w == "foreign_writes") return g_foreign_writes;
    if (w == "writes_while_busy") return g_writes_while_busy;
    if (w == "capture_broken") return g_capture_broken;
    if (w == "last_error") return g_last;
    return -1;
}

// ---- the runtime's side
cudaError_t cudaMalloc(void **p, size_t n) {
    *p = nullptr;
    if (g_forbid_malloc) return ret(cudaErrorStreamCaptureUnsupported);
    if (fails() || g_live_bytes + n > g_limit) return ret(cudaErrorMemoryAllocation);
    *p = malloc(n);
    g_live[*p] = {n, g_current};
    g_live_bytes += n;
    ++g_mallocs;
    return cudaSuccess;
}
cudaError_t cudaFree(void *p) {
    if (!p) return cudaSuccess;
    auto it = g_live.find(p);
    if (it == g_live.end()) return ++g_foreign_frees, ret(cudaErrorInvalidValue);
    g_busy = false;               // waits for the device
    g_live_bytes -= it->second.bytes;
    g_live.erase(it);
    free(p);
    ++g_frees;
    return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void *dst, const void *src, size_t n, cudaMemcpyKind kind, cudaStream_t) {
    if (kind == cudaMemcpyDeviceToHost) return cudaSuccess;
    auto it = g_live.upper_bound(dst);
    if (it == g_live.begin()) return ++g_foreign_writes, cudaSuccess;
    --it;
    if (static_cast<char *>(dst) + n > static_cast<char *>(it->first) + it->second.bytes || it->second.context != g_current) return ++g_foreign_writes, cudaSuccess;
    g_writes_while_busy += g_busy;
    memcpy(dst, src, n);
    return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void *p, int, size_t, cudaStream_t) { return g_foreign_writes += g_live.count(p) == 0, cudaSuccess; }
cudaError_t cudaDeviceSynchronize() {
    if (g_capture_elsewhere) return g_capture_broken = true, ret(cudaErrorStreamCaptureUnsupported);
    g_busy = false;
    return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus *s) { return *s = cudaStreamCaptureStatusNone, cudaSuccess; }
cudaError_t cudaGetDevice(int *d) { return *d = 0, cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr, int) { return *v = 148, cudaSuccess; }
cudaError_t cudaGetLastError() {
    const cudaError_t e = g_last;
    g_last = cudaSuccess;
    return e;
}
const char *cudaGetErrorName(cudaError_t) { return "fake"; }
const char *cudaGetErrorString(cudaError_t) { return "fake"; }
cudaError_t cudaGetDriverEntryPoint(const char *name, void **fn, unsigned long long, cudaDriverEntryPointQueryResult *q) {
    const std::string n = name;
    *fn = n == "cuCtxGetId"                  ? reinterpret_cast<void *>(get_id)
          : n == "cuDevicePrimaryCtxGetState" ? reinterpret_cast<void *>(get_state)
          : n == "cuDevicePrimaryCtxRetain"  ? reinterpret_cast<void *>(retain)
          : n == "cuDevicePrimaryCtxRelease" ? reinterpret_cast<void *>(release)
          : n == "cuDeviceGet"               ? reinterpret_cast<void *>(get_device)
                                             : nullptr;
    *q = *fn ? cudaDriverEntryPointSuccess : cudaDriverEntryPointSymbolNotFound;
    return cudaSuccess;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) { return fails() ? ret(cudaErrorUnknown) : (*s = reinterpret_cast<cudaStream_t>(new char), cudaSuccess); }
cudaError_t cudaStreamDestroy(cudaStream_t s) { return delete reinterpret_cast<char *>(s), cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t e, unsigned) { return e ? cudaSuccess : ret(cudaErrorInvalidResourceHandle); }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) { return fails() ? ret(cudaErrorUnknown) : (*e = reinterpret_cast<cudaEvent_t>(new char), cudaSuccess); }
cudaError_t cudaEventDestroy(cudaEvent_t e) { return delete reinterpret_cast<char *>(e), cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t) { return e ? cudaSuccess : ret(cudaErrorInvalidResourceHandle); }

}  // extern "C"

namespace tessera {
cudaError_t launch_gather(const tessera_plan *, const void *, const void *, void *, void *, GatherMode, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_kv_fp8(const tessera_plan *, const void *, const void *, void *, void *, bool, bool, float, float, cudaStream_t) { abort(); }
cudaError_t launch_scatter_fresh(const tessera_plan *, void *, void *, const void *, const void *, int, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_rope_fresh(const tessera_plan *, void *, void *, cudaStream_t) { abort(); }
cudaError_t launch_extend_write(const tessera_plan *, void *, void *, void *, const void *, const void *, void *, void *, cudaStream_t) { abort(); }
cudaError_t launch_attn_tc(const tessera_plan *, void *, void *, const void *, void *, float *, int, int, cudaStream_t, std::string *) { return cudaSuccess; }
cudaError_t launch_attn_tc_k8(const tessera_plan *, void *, void *, const void *, void *, float *, float, cudaStream_t, std::string *) { abort(); }
cudaError_t launch_compose_k8(const tessera_plan *, const void *, const void *, void *, void *, bool, float, cudaStream_t) { abort(); }
cudaError_t launch_fresh_k8(const tessera_plan *, const void *, void *, float, void *, void *, const void *, const void *, float, cudaStream_t) { abort(); }
}  // namespace tessera
