#include "blob_pool.h"

#include <mutex>

#include <cuda.h>

namespace tessera {

namespace {

constexpr int kMaxDevices = 64;
constexpr size_t kGuardBytes = 256;

// A fixed array: nothing here allocates host memory, so nothing throws through the C entry points.
struct Pool {
    std::mutex mutex;
    unsigned long long context = 0;    // id of the primary context the blocks belong to
    void *anchor = nullptr;            // keeps the driver's slab of small allocations mapped: beside it a guard's cudaMalloc
                                       // and cudaFree take 2.1 + 3.4 us, alone in its slab 700 + 570 and more
    DeviceBlob blocks[kBlobPoolBlocks];     // oldest first
    int count = 0;
    size_t held = 0;

    DeviceBlob take(int i) {
        const DeviceBlob b = blocks[i];
        for (int k = i; k + 1 < count; ++k) blocks[k] = blocks[k + 1];
        --count;
        held -= b.bytes;
        return b;
    }
    // A device has one primary context at a time: blocks of an earlier one went with the reset that ended it.
    void enter(unsigned long long id) {
        if (context == id) return;
        context = id;
        anchor = nullptr;
        count = 0;
        held = 0;
    }
};
Pool g_pools[kMaxDevices];

template <class Fn>
Fn driver_fn(const char *name) {
    void *p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint(name, &p, cudaEnableDefault, &q) != cudaSuccess || q != cudaDriverEntryPointSuccess) p = nullptr;
    return reinterpret_cast<Fn>(p);
}

// Id of a context (null: the current one; ids are never used twice in a process), 0 when there is none.
unsigned long long context_id(CUcontext c = nullptr) {
    static const auto get_id = driver_fn<CUresult (*)(CUcontext, unsigned long long *)>("cuCtxGetId");
    unsigned long long id = 0;
    return get_id && get_id(c, &id) == CUDA_SUCCESS ? id : 0;
}

// Id of the primary context of `device`, 0 when it has none (and none is made).
unsigned long long primary_context_id(int device) {
    static const auto get_device = driver_fn<CUresult (*)(CUdevice *, int)>("cuDeviceGet");
    static const auto get_state = driver_fn<CUresult (*)(CUdevice, unsigned *, int *)>("cuDevicePrimaryCtxGetState");
    static const auto retain = driver_fn<CUresult (*)(CUcontext *, CUdevice)>("cuDevicePrimaryCtxRetain");
    static const auto release = driver_fn<CUresult (*)(CUdevice)>("cuDevicePrimaryCtxRelease");
    CUdevice dev;
    CUcontext primary = nullptr;
    unsigned flags = 0;
    int active = 0;
    if (device < 0 || device >= kMaxDevices || !get_device || !get_state || !retain || !release) return 0;
    if (get_device(&dev, device) != CUDA_SUCCESS || get_state(dev, &flags, &active) != CUDA_SUCCESS || !active) return 0;
    if (retain(&primary, dev) != CUDA_SUCCESS) return 0;
    const unsigned long long id = context_id(primary);
    release(dev);
    return id;
}

}  // namespace

cudaError_t blob_acquire(DeviceBlob *b, size_t bytes, cudaStream_t stream) {
    int device = 0;
    cudaError_t e = cudaGetDevice(&device);
    if (e != cudaSuccess) return e;
    // sizes in steps of an eighth: plans of about the same size fit each other's blocks
    size_t step = 4096;
    while (step * 8 < bytes) step *= 2;
    bytes = (bytes + step - 1) / step * step;
    if (context_id() == 0) cudaFree(nullptr);          // the first call of the process: makes the primary context
    // A captured copy belongs to a graph that may run after the plan is gone: it gets memory that is never pooled.
    cudaStreamCaptureStatus capturing = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(stream, &capturing) != cudaSuccess) {
        cudaGetLastError();
        capturing = cudaStreamCaptureStatusActive;
    }
    const unsigned long long context = capturing == cudaStreamCaptureStatusNone ? context_id() : 0;
    Pool &pl = g_pools[device < kMaxDevices ? device : 0];
    std::unique_lock<std::mutex> lock(pl.mutex);
    // (a context that was the primary one stays it while it lives: asked once per context)
    if (context == 0 || device >= kMaxDevices || (context != pl.context && context != primary_context_id(device))) {
        lock.unlock();
        void *p = nullptr;
        if ((e = cudaMalloc(&p, bytes)) == cudaSuccess) *b = {p, bytes, device, 0, nullptr};
        return e;
    }
    pl.enter(context);
    auto allocate = [&pl](void **p, size_t n) {
        cudaError_t r = cudaMalloc(p, n);
        while (r == cudaErrorMemoryAllocation && pl.count > 0) {
            if (cudaFree(pl.take(0).p) != cudaSuccess) continue;
            cudaGetLastError();
            r = cudaMalloc(p, n);
        }
        return r;
    };
    if (!pl.anchor && (e = allocate(&pl.anchor, kGuardBytes)) != cudaSuccess) return e;
    void *guard = nullptr;
    if ((e = allocate(&guard, kGuardBytes)) != cudaSuccess) return e;
    int best = -1;
    for (int i = 0; i < pl.count; ++i) {
        if (pl.blocks[i].bytes < bytes || pl.blocks[i].bytes > 2 * bytes) continue;
        if (best < 0 || pl.blocks[i].bytes < pl.blocks[best].bytes) best = i;
    }
    void *p = nullptr;
    if (best >= 0) {
        *b = pl.take(best);
    } else if ((e = allocate(&p, bytes)) == cudaSuccess) {
        *b = {p, bytes, device, context, nullptr};
    } else {
        cudaFree(guard);
        return e;
    }
    b->guard = guard;
    return cudaSuccess;
}

cudaError_t blob_release(const DeviceBlob &b) {
    if (b.context == 0) return cudaFree(b.p);
    const bool current = context_id() == b.context;
    if (!current && primary_context_id(b.device) != b.context) return cudaErrorContextIsDestroyed;   // freed by a reset
    cudaError_t e = cudaFree(b.guard);                  // waits for the device
    if (e != cudaSuccess || !current || b.bytes > kBlobPoolBytes) {
        const cudaError_t f = cudaFree(b.p);
        return e != cudaSuccess ? e : f;
    }
    Pool &pl = g_pools[b.device];
    std::lock_guard<std::mutex> lock(pl.mutex);
    pl.enter(b.context);
    while (pl.count == kBlobPoolBlocks || (pl.count > 0 && pl.held + b.bytes > kBlobPoolBytes)) {
        const cudaError_t f = cudaFree(pl.take(0).p);
        if (e == cudaSuccess) e = f;
    }
    pl.blocks[pl.count++] = b;
    pl.held += b.bytes;
    return e;
}

}  // namespace tessera
