#include "blob_pool.h"

#include <deque>
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

struct Pool {
    std::mutex mutex;
    std::deque<Block> blocks;     // oldest first
    size_t held = 0;
};

Pool &pool() {
    static Pool *p = new Pool;    // never destroyed: the driver may be gone before static destructors run
    return *p;
}

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
Block take(Pool &pl, size_t i) {
    const Block b = pl.blocks[i];
    pl.blocks.erase(pl.blocks.begin() + (std::ptrdiff_t)i);
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
    Pool &pl = pool();
    std::lock_guard<std::mutex> lock(pl.mutex);
    if (capturing == cudaStreamCaptureStatusNone) {
        size_t best = pl.blocks.size();
        for (size_t i = 0; i < pl.blocks.size(); ++i) {
            const Block &b = pl.blocks[i];
            if (b.device != device || b.context != context || b.bytes < bytes || b.bytes > 2 * bytes) continue;
            if (best == pl.blocks.size() || b.bytes < pl.blocks[best].bytes) best = i;
        }
        if (best < pl.blocks.size()) {
            const Block b = take(pl, best);
            *p = b.p;
            *granted = b.bytes;
            return cudaSuccess;
        }
    }
    e = cudaMalloc(p, bytes);
    if (e == cudaErrorMemoryAllocation) {
        bool any = false;
        for (size_t i = pl.blocks.size(); i-- > 0;)
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
        Pool &pl = pool();
        std::lock_guard<std::mutex> lock(pl.mutex);
        pl.blocks.push_back({p, bytes, device, context});
        pl.held += bytes;
        while (pl.held > kBlobPoolBytes) {
            const Block b = take(pl, 0);
            if (b.device != device) cudaSetDevice(b.device);
            if (context_id() == b.context) {
                const cudaError_t f = cudaFree(b.p);
                if (e == cudaSuccess) e = f;
            }
            if (b.device != device) cudaSetDevice(device);
        }
    }
    if (current != device) cudaSetDevice(current);
    return e;
}

}  // namespace tessera
