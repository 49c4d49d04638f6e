// Device memory of plans.  A plan is created and destroyed per batch, and cudaMalloc / cudaFree of its tables and
// split-KV workspace (0.3 MB and 11 MB for one 5 312-token request) cost several times what building the plan
// costs, so blocks of destroyed plans are kept for the next ones.  So do the 8-bit copy of q and the staging buffers,
// which a plan's first call asks for.
#pragma once
#include <cstddef>

#include <cuda_runtime.h>

namespace tessera {

// Per device: room for the largest block a plan asks for.  Split-KV of up to four rounds of attention items takes up to
// 16 x SMs slots of 66 560 bytes (158 MB on 148 SMs, head_dim 128), and a block that is not kept costs 0.7 ms of
// cudaMalloc + cudaFree per plan: ten prompts of 12 288 tokens (51 MB), plan and one layer 2 370 -> 1 640 us.
constexpr size_t kBlobPoolBytes = size_t(192) << 20;
constexpr int kBlobPoolBlocks = 16;

struct DeviceBlob {
    void *p = nullptr;
    size_t bytes = 0;
    int device = -1;
    unsigned long long context = 0;    // id of the context it was allocated in; 0: never pooled
    void *guard = nullptr;             // of a block that may be pooled: a few bytes allocated and freed with every plan
};

// A block of at least `bytes` on the current device.  Refused whenever cudaMalloc is (a capture that forbids it on
// any stream), also when a kept block would do; not pooled when `stream` itself is being captured.  Thread-safe.
cudaError_t blob_acquire(DeviceBlob *b, size_t bytes, cudaStream_t stream);

// Returns a block once all work of its device has ended: the guard's cudaFree waits for it, and is allowed wherever
// the plan's own cudaFree would be (cudaDeviceSynchronize is not: it breaks every capture of the context, thread-local
// and relaxed ones on other threads too).  At most kBlobPoolBytes in
// kBlobPoolBlocks blocks stay in a device's pool (the oldest go first); when an allocation fails all are given back.
// Only blocks of a device's primary context are kept, and only while that context is the current one; anything else
// is a plain cudaFree.
cudaError_t blob_release(const DeviceBlob &b);

}  // namespace tessera
