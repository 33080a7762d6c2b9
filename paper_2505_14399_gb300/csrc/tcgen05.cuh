// The fifth-generation tensor core as inline PTX: accumulator (tensor memory) allocation, shared
// memory matrix descriptors, the fp16 MMA, its completion barrier, accumulator loads.
#pragma once

#include <cstdint>

#include "tma.cuh"

namespace wmg {

// ---- tensor memory: 128 lanes x `cols` 32-bit columns (a power of two, at least 32); one warp.
// An allocation waits while other CTAs of the SM hold the columns, and ends with them.
__device__ __forceinline__ void tc5_alloc(uint32_t* dst, uint32_t cols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                   smem_addr(dst)),
               "r"(cols)
               : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tc5_dealloc(uint32_t tmem, uint32_t cols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(cols)
               : "memory");
}

// order tensor-core operations of this thread against a thread barrier before / after it
__device__ __forceinline__ void tc5_fence_before() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc5_fence_after() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}

// Shared memory matrix descriptor without swizzle, for MN-major operands: core matrices of eight
// k rows of eight 16-bit columns (128 contiguous bytes), `kstride` bytes between octets of k,
// `mnstride` between octets of columns.  All multiples of 16 bytes.
__device__ __forceinline__ uint64_t tc5_desc(uint32_t addr, uint32_t kstride, uint32_t mnstride) {
  return (uint64_t)((addr >> 4) & 0x3fffu) | ((uint64_t)((kstride >> 4) & 0x3fffu) << 16) |
         ((uint64_t)((mnstride >> 4) & 0x3fffu) << 32) | (1ull << 46);
}

// Instruction descriptor: FP32 accumulators, fp16 A and B, both MN-major, M rows, N columns (N
// may be or-ed in later)
__host__ __device__ constexpr uint32_t tc5_idesc_n(int n) { return (uint32_t)(n >> 3) << 17; }
__host__ __device__ constexpr uint32_t tc5_idesc_f16_mn(int m, int n) {
  return (1u << 4) | (1u << 15) | (1u << 16) | tc5_idesc_n(n) |
         ((uint32_t)(m >> 4) << 24);
}

// D (+)= A B, K = 16, issued by one thread; acc 0 overwrites D
__device__ __forceinline__ void tc5_mma(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc,
                                        uint32_t acc) {
  asm volatile(
      "{\n"
      " .reg .pred p;\n"
      " setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n"
      "}\n" ::"r"(d),
      "l"(a), "l"(b), "r"(idesc), "r"(acc)
      : "memory");
}
// one arrival on `bar` when this thread's earlier MMAs have completed
__device__ __forceinline__ void tc5_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                   smem_addr(bar))
               : "memory");
}

// four consecutive accumulator columns of this warp's 32 lanes (lane 32 (warp % 4) + lane)
__device__ __forceinline__ void tc5_ld4(float v[4], uint32_t addr) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
               : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3])
               : "r"(addr)
               : "memory");
}
__device__ __forceinline__ void tc5_wait_ld() {
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

}  // namespace wmg
