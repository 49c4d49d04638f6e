// Global-memory accesses and grid-dependency instructions shared by the kernels.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

namespace tessera {

// Programmatic dependent launch: a kernel started through launch_kernel(.., chained = true) may be resident while
// its predecessor in the stream still runs.  grid_wait() returns once every preceding grid has completed and its
// writes are visible; every kernel launched that way calls it in all threads (so a grid's completion implies its
// predecessors') before its first access to anything a kernel may have written.  The plan's tables are not among
// that: they were copied before the first launch of the plan, and a chained kernel waits for copies and events
// like any other.  grid_release() lets the successor's blocks take the
// room that this grid's last wave leaves.
__device__ __forceinline__ void grid_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_release() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Read-once data.  Not the non-coherent path: a chained kernel's lifetime overlaps the kernel that wrote them.
__device__ __forceinline__ uint4 ldg_stream(const uint4 *p) {
    uint4 v;
    asm volatile("ld.global.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p) : "memory");
    return v;
}
// Rows read once, but in pieces of less than a 128-byte line per instruction (8-bit codes: the two halves of a head are
// 64 bytes each, 32 at head_dim 64): the line stays in L1 until its other pieces have been read, so that the host link
// is asked for whole lines.  65 536 rows of codes out of pinned memory: L1::no_allocate 3.19 ms, so 2.62 (head_dim 64:
// 2.62 and 1.35); 16-bit rows of head_dim 64 in device memory, rounded to codes: plain loads 43.4 us, so 40.4.  Whole
// lines are better off without: 16-bit rows of head_dim 128 to codes 86.3 us, L1::no_allocate 85.9.
__device__ __forceinline__ uint2 ldg_pieces(const uint2 *p) {
    uint2 v;
    asm volatile("ld.global.L1::evict_first.v2.u32 {%0,%1}, [%2];" : "=r"(v.x), "=r"(v.y) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ uint4 ldg_pieces(const uint4 *p) {
    uint4 v;
    asm volatile("ld.global.L1::evict_first.v4.u32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ uint4 ldg_plain(const uint4 *p) {
    uint4 v;
    asm volatile("ld.global.v4.u32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void stg(uint4 *p, const uint4 &v) {
    asm volatile("st.global.v4.u32 [%0], {%1,%2,%3,%4};" ::"l"(p), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}

}  // namespace tessera
