// bulkcopy.cuh -- asynchronous copy primitives (inline PTX) of the kernels that
// bring global memory to shared memory or to L2 ahead of its use.
#pragma once
#include "modarith.cuh"

namespace he {

__device__ __forceinline__ u32 bc_smem(const void *p) { return (u32)__cvta_generic_to_shared(p); }

// 16 bytes from global `src` to shared address `dst` (both 16-byte aligned),
// through L2 only.
__device__ __forceinline__ void bc_copy16(u32 dst, const void *src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
// Closes a group (possibly empty) of this thread's copies.
__device__ __forceinline__ void bc_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
// Waits until at most the LEFT newest groups of this thread are under way.
template <int LEFT>
__device__ __forceinline__ void bc_wait_groups() {
    asm volatile("cp.async.wait_group %0;" ::"n"(LEFT) : "memory");
}

// Asks the copy engine to bring `bytes` (a multiple of 16, 16-byte aligned)
// of global memory into L2; nothing waits for it.
__device__ __forceinline__ void bc_prefetch_l2(const void *src, u32 bytes) {
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(src), "r"(bytes) : "memory");
}

}  // namespace he
