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
__device__ __forceinline__ uint2 ldg_stream(const uint2 *p) {
    uint2 v;
    asm volatile("ld.global.L1::no_allocate.v2.u32 {%0,%1}, [%2];" : "=r"(v.x), "=r"(v.y) : "l"(p) : "memory");
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
