// tcgen05 / mbarrier helpers of the contractions (digit_gemm.cuh).
#pragma once
#include "kernels_common.cuh"

namespace mdp {

constexpr long long TC_WAIT_CYCLES = 4000000000LL;   // limit of every wait, about 2 s at the maximum clock

__device__ __forceinline__ uint64_t smem_desc(unsigned addr, unsigned lbo, unsigned sbo) {
  // shared-memory matrix descriptor: start address, leading (K) and stride (M/N) byte offsets of
  // the 8 x 16-byte core matrices, descriptor version 1, no swizzle
  return (uint64_t)((addr >> 4) & 0x3FFF) | ((uint64_t)((lbo >> 4) & 0x3FFF) << 16) |
         ((uint64_t)((sbo >> 4) & 0x3FFF) << 32) | ((uint64_t)1 << 46);
}
// instruction descriptor of kind::f16: FP32 accumulator, fp16 A and B, both K-major, M = 128
__host__ __device__ constexpr uint32_t f16_idesc(uint32_t n) { return (1u << 4) | ((n >> 3) << 17) | ((128u >> 4) << 24); }

__device__ __forceinline__ bool mbar_try(unsigned addr, unsigned parity) {
  unsigned ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok) : "r"(addr), "r"(parity) : "memory");
  return ok != 0;
}
// wait for the completion of the phase with parity `parity`, at most TC_WAIT_CYCLES; false when
// the limit ran out or another warp has already given up (*abort)
__device__ __forceinline__ bool mbar_wait(unsigned addr, unsigned parity, volatile int *abort) {
  const long long t0 = clock64();
  while (!mbar_try(addr, parity)) {
    if (*abort) return false;
    if (clock64() - t0 > TC_WAIT_CYCLES) { *abort = 1; return false; }
  }
  return true;
}
__device__ __forceinline__ void mbar_arrive(unsigned addr) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(addr) : "memory");
}
__device__ __forceinline__ void mbar_init(unsigned addr, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(addr), "r"(count) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_commit(unsigned mbar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(mbar) : "memory");
}
// D (tensor memory) = A B (+ D when acc), kind::f16, operands in shared memory
__device__ __forceinline__ void tc_mma(unsigned d, uint64_t da, uint64_t db, uint32_t idesc, unsigned acc) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d), "l"(da), "l"(db), "r"(idesc), "r"(acc)
      : "memory");
}

// two fp16 digits in one word: byte K (0 = least significant) of the values a (low half) and b
// (high half), each under the fp16 exponent of 1024, minus 1024 + 128 (exact)
template <int K>
__device__ __forceinline__ unsigned digit_pair(unsigned ahi, unsigned alo, unsigned bhi, unsigned blo) {
  constexpr unsigned k = K & 3;
  constexpr unsigned sel = k | (k << 4) | ((4 + k) << 8) | ((4 + k) << 12);
  const unsigned w = __byte_perm(K >= 4 ? ahi : alo, K >= 4 ? bhi : blo, sel);
  unsigned r;
  asm("{\n .reg .b32 t;\n lop3.b32 t, %1, %2, %3, 0xEA;\n sub.rn.f16x2 %0, t, %4;\n}\n"
      : "=r"(r) : "r"(w), "r"(0x00FF00FFu), "r"(0x64006400u), "r"(0x64806480u));
  return r;
}

}  // namespace mdp
