// Device memory of plans.  A plan is created and destroyed per batch, and cudaMalloc / cudaFree of its tables and
// split-KV workspace (0.3 MB and 11 MB for one 5 312-token request) cost several times what building the plan
// costs, so blocks of destroyed plans are kept for the next ones.
#pragma once
#include <cstddef>

#include <cuda_runtime.h>

namespace tessera {

constexpr size_t kBlobPoolBytes = size_t(64) << 20;
constexpr int kBlobPoolBlocks = 16;

// A block of at least `bytes` on the current device (`*granted`: its size).  Refused, like cudaMalloc, while
// `stream` is being captured.  Thread-safe.
cudaError_t blob_acquire(void **p, size_t bytes, size_t *granted, cudaStream_t stream);

// Returns a block of `device` after waiting, as cudaFree does, for all work of that device.  At most kBlobPoolBytes
// in kBlobPoolBlocks blocks stay in the pool over all devices (the oldest go first); when an allocation fails everything is given back.
cudaError_t blob_release(void *p, size_t bytes, int device);

}  // namespace tessera
