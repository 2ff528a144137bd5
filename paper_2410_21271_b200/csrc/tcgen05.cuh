// Instructions of the 5th-generation tensor cores that more than one kernel family issues.
#pragma once
#include "decode_common.cuh"

namespace eora {
namespace dec {

// D += A B^T, both operands in shared memory and of the same 16-bit type (which one idesc says).
__device__ __forceinline__ void umma_f16(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t accumulate) {
  asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\ttcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
               ::"r"(tmem_d), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate) : "memory");
}
// Arrives at the barrier when the MMAs that this thread has issued have completed.
__device__ __forceinline__ void umma_commit_a(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void umma_commit(uint64_t* bar) { umma_commit_a(smem_u32(bar)); }
__device__ __forceinline__ bool elect_one() {
  uint32_t p;
  asm volatile("{\n\t.reg .pred q;\n\telect.sync _|q, 0xffffffff;\n\tselp.u32 %0, 1, 0, q;\n\t}" : "=r"(p));
  return p != 0;
}
// K-major operand descriptor for rows of BYTES (64 or 128) swizzled over as many, 8-row groups 8 BYTES apart.
template <int BYTES>
__device__ __forceinline__ uint64_t make_desc(uint32_t addr) {
  static_assert(BYTES == 64 || BYTES == 128, "the swizzles in use");
  const uint32_t lo = ((addr & 0x3FFFFu) >> 4) | (1u << 16);            // start address, leading byte offset (unused) = 1
  const uint32_t hi = (8 * BYTES) >> 4 | (1u << 14) | (BYTES == 128 ? 2u : 4u) << 29;      // stride byte offset, descriptor version 1, swizzle
  return ((uint64_t)hi << 32) | lo;
}

}  // namespace dec
}  // namespace eora
