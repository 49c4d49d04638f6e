// Launch entry points of the individual kernels (internal to the library).
#pragma once
#include <cuda_runtime.h>

#include "plan.h"

namespace tessera {

enum class GatherMode { kCopy, kCopyRotate, kShiftInPlace };

void count_launch();   // bumps the process-wide kernel-launch counter

// Launches and counts `kernel`.  `chained`: it may become resident while its predecessor in the stream still runs
// (the kernel itself waits, see grid_wait()); behind anything but a kernel that is an ordinary launch too.
// `cluster`: thread blocks per cluster (2: blocks 2 i and 2 i + 1 run on the two SMs of one TPC).
template <class... P, class... A>
cudaError_t launch_clusters(void (*kernel)(P...), unsigned grid, unsigned block, unsigned cluster, size_t smem, cudaStream_t st,
                            bool chained, A... args) {
    cudaLaunchAttribute attr[2]{};
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = attr;
    if (chained) {
        attr[cfg.numAttrs].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[cfg.numAttrs++].val.programmaticStreamSerializationAllowed = 1;
    }
    if (cluster > 1) {
        attr[cfg.numAttrs].id = cudaLaunchAttributeClusterDimension;
        attr[cfg.numAttrs].val.clusterDim.x = cluster;
        attr[cfg.numAttrs].val.clusterDim.y = attr[cfg.numAttrs].val.clusterDim.z = 1;
        ++cfg.numAttrs;
    }
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
    if (e == cudaSuccess) count_launch();
    else cudaGetLastError();          // returned here, not left for a later call's own check
    return e;
}
template <class... P, class... A>
cudaError_t launch_kernel(void (*kernel)(P...), unsigned grid, unsigned block, size_t smem, cudaStream_t st, bool chained, A... args) {
    return launch_clusters(kernel, grid, block, 1, smem, st, chained, args...);
}

// Sources are read from (k_src, v_src) - the destination pools themselves unless the plan names a
// separate source pool - and written to the plan's destination slots in (k_pool, v_pool).
cudaError_t launch_gather(const tessera_plan *pl, const void *k_src, const void *v_src, void *k_pool, void *v_pool,
                          GatherMode mode, cudaStream_t st);
// Host-tier readers over gather runs [first_run, first_run + n_runs): every source row is read once and written
// to the slots of all its users, keys rotated; 16-bit, respectively e4m3, sources.  max_blocks > 0 caps the
// grid: the blocks then walk the runs, so the launch occupies only a few SMs beside the attention kernel.
cudaError_t launch_gather_runs(const tessera_plan *pl, const void *k_src, const void *v_src, void *k_pool, void *v_pool,
                               int first_run, int n_runs, int max_blocks, cudaStream_t st);
cudaError_t launch_expand_fp8_runs(const tessera_plan *pl, const void *k_src8, const void *v_src8, void *k_pool, void *v_pool,
                                   float k_scale, float v_scale, int first_run, int n_runs, int max_blocks, cudaStream_t st);
// 8-bit (e4m3) tier.  to_8bit false: (k_src, v_src) hold codes, (k_dst, v_dst) 16-bit pages, mul = scale;
// to_8bit true: the reverse, mul = 1 / scale.  Copy list and shift table are the plan's.
cudaError_t launch_kv_fp8(const tessera_plan *pl, const void *k_src, const void *v_src, void *k_dst, void *v_dst,
                          bool to_8bit, bool rotate, float k_mul, float v_mul, cudaStream_t st);
// In-place rotation of the fresh q / k_new rows for their target positions (either may be null).
cudaError_t launch_rope_fresh(const tessera_plan *pl, void *q, void *k_new, cudaStream_t st);
// Fused write side of the extend pass: rotate q in place, write rotated K / V rows to their slots and raw
// K / V rows of captured units to their cache slots (k_cache / v_cache may be null when nothing is captured).
cudaError_t launch_extend_write(const tessera_plan *pl, void *k_pool, void *v_pool, void *q, const void *k_new_raw,
                                const void *v_new, void *k_cache, void *v_cache, cudaStream_t st);
// chunk < 0: the whole batch; otherwise only request chunk `chunk` (see tessera_plan::chunk_row_off).
// k_new / v_new / q / out / lse always point at row 0 of the whole batch.
cudaError_t launch_scatter_fresh(const tessera_plan *pl, void *k_pool, void *v_pool, const void *k_new,
                                 const void *v_new, int chunk, cudaStream_t st);
// tcgen05 attention; returns cudaErrorNotSupported when the plan's shape is outside its range (the plan
// builder accepts no such shape).
// max_blocks > 0 caps the persistent grid below one block per SM (SMs left to a concurrent reader kernel); refused where
// the whole list has more items than SMs, because it is dealt out for the full grid.
cudaError_t launch_attn_tc(const tessera_plan *pl, void *k_pool, void *v_pool, const void *q, void *out,
                           float *lse, int chunk, int max_blocks, cudaStream_t st, std::string *err);

// The same kernel with 8-bit (e4m3) queries and keys: q8 [n_q][H_q][D] and k_pool8 hold codes, qk_scale is the
// product of their two scales; head_dim 128 only; the whole batch on the full grid.
cudaError_t launch_attn_tc_k8(const tessera_plan *pl, void *k_pool8, void *v_pool, const void *q8, void *out,
                              float *lse, float qk_scale, cudaStream_t st, std::string *err);
// Compose for the 8-bit-key attention path: 16-bit sources -> keys (rotated, times k_mul) as e4m3 codes in
// k_dst8, values as bit copies in the 16-bit v_dst.
cudaError_t launch_compose_k8(const tessera_plan *pl, const void *k_src, const void *v_src, void *k_dst8, void *v_dst,
                              bool rotate, float k_mul, cudaStream_t st);
// Fresh rows of the 8-bit-key path: q -> e4m3 codes of (q * q_mul) in q8, k_new / v_new (null: skipped) into an 8-bit
// key pool (codes of k_new * k_mul; nearest-even, saturating) and a 16-bit value pool (bit copies).
cudaError_t launch_fresh_k8(const tessera_plan *pl, const void *q, void *q8, float q_mul, void *k_pool8, void *v_pool,
                            const void *k_new, const void *v_new, float k_mul, cudaStream_t st);

}  // namespace tessera
