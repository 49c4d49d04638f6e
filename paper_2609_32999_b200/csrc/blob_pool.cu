#include "blob_pool.h"

#include <mutex>

#include <cuda.h>

namespace tessera {

namespace {

struct Block {
    void *p;
    size_t bytes;
    int device;
    unsigned long long context;   // id of the context the block belongs to: a block does not outlive a device reset
};

// A fixed array: nothing here allocates host memory, so nothing throws through the C entry points.
struct Pool {
    std::mutex mutex;
    Block blocks[kBlobPoolBlocks];     // oldest first
    int count = 0;
    size_t held = 0;
};
Pool g_pool;

// Id of the current context, 0 when it cannot be asked for (then nothing is pooled).
unsigned long long context_id() {
    using Fn = CUresult (*)(CUcontext, unsigned long long *);
    static const Fn fn = [] {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuCtxGetId", &p, cudaEnableDefault, &q) != cudaSuccess || q != cudaDriverEntryPointSuccess) p = nullptr;
        return reinterpret_cast<Fn>(p);
    }();
    unsigned long long id = 0;
    return fn && fn(nullptr, &id) == CUDA_SUCCESS ? id : 0;
}

// Takes block i out of the pool.
Block take(Pool &pl, int i) {
    const Block b = pl.blocks[i];
    for (int k = i; k + 1 < pl.count; ++k) pl.blocks[k] = pl.blocks[k + 1];
    --pl.count;
    pl.held -= b.bytes;
    return b;
}

}  // namespace

cudaError_t blob_acquire(void **p, size_t bytes, size_t *granted, cudaStream_t stream) {
    cudaStreamCaptureStatus capturing = cudaStreamCaptureStatusNone;
    cudaError_t e = cudaStreamIsCapturing(stream, &capturing);
    if (e != cudaSuccess) return e;
    int device = 0;
    if ((e = cudaGetDevice(&device)) != cudaSuccess) return e;
    // sizes in steps of an eighth: plans of about the same size fit each other's blocks
    size_t step = 4096;
    while (step * 8 < bytes) step *= 2;
    bytes = (bytes + step - 1) / step * step;
    const unsigned long long context = context_id();
    Pool &pl = g_pool;
    std::lock_guard<std::mutex> lock(pl.mutex);
    if (capturing == cudaStreamCaptureStatusNone) {
        int best = -1;
        for (int i = 0; i < pl.count; ++i) {
            const Block &b = pl.blocks[i];
            if (b.device != device || b.context != context || b.bytes < bytes || b.bytes > 2 * bytes) continue;
            if (best < 0 || b.bytes < pl.blocks[best].bytes) best = i;
        }
        if (best >= 0) {
            const Block b = take(pl, best);
            *p = b.p;
            *granted = b.bytes;
            return cudaSuccess;
        }
    }
    e = cudaMalloc(p, bytes);
    if (e == cudaErrorMemoryAllocation) {
        bool any = false;
        for (int i = pl.count; i-- > 0;)
            if (pl.blocks[i].device == device) {
                const Block b = take(pl, i);
                if (b.context == context) any |= cudaFree(b.p) == cudaSuccess;
            }
        if (any) {
            cudaGetLastError();
            e = cudaMalloc(p, bytes);
        }
    }
    *granted = bytes;
    return e;
}

cudaError_t blob_release(void *p, size_t bytes, int device) {
    int current = 0;
    cudaError_t e = cudaGetDevice(&current);
    if (e == cudaSuccess && current != device) e = cudaSetDevice(device);
    if (e != cudaSuccess) return e;
    const unsigned long long context = context_id();
    if (context == 0 || bytes > kBlobPoolBytes / 2) {
        e = cudaFree(p);
    } else if ((e = cudaDeviceSynchronize()) != cudaSuccess) {
        cudaFree(p);
    } else {
        Pool &pl = g_pool;
        std::lock_guard<std::mutex> lock(pl.mutex);
        while (pl.count == kBlobPoolBlocks || (pl.count > 0 && pl.held + bytes > kBlobPoolBytes)) {
            const Block b = take(pl, 0);
            if (b.device != device) cudaSetDevice(b.device);
            if (context_id() == b.context) {
                const cudaError_t f = cudaFree(b.p);
                if (e == cudaSuccess) e = f;
            }
            if (b.device != device) cudaSetDevice(device);
        }
        pl.blocks[pl.count++] = {p, bytes, device, context};
        pl.held += bytes;
    }
    if (current != device) cudaSetDevice(current);
    return e;
}

}  // namespace tessera
