// sfm_umma.cuh -- mbarriers and 5th-generation tensor-core products, shared by
// the field product (sfm_product.cu) and the surrogate's convolution
// (sfm_surrogate.cu).
#pragma once
#include "sfm_device.cuh"

namespace sfm {

// Bounded wait for the mbarrier phase `parity`; false when it ran out.  The
// bound is about a second of the global timer, with an iteration cap behind it.
__device__ __forceinline__ bool mbar_wait(uint32_t mbar, uint32_t parity) {
  unsigned long long t0 = 0;
  for (int it = 0; it < (1 << 26); ++it) {
    uint32_t done = 0;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}\n"
        : "=r"(done)
        : "r"(mbar), "r"(parity)
        : "memory");
    if (done) return true;
    if (second_is_over(it, t0)) return false;
  }
  return false;
}

__device__ __forceinline__ void mbar_arrive(uint32_t mbar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(mbar) : "memory");
}

// shared-memory matrix descriptor, no swizzle: start, K-direction (leading)
// and M/N-direction (stride) byte offsets between core matrices
__device__ __forceinline__ uint64_t umma_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
  return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)(lbo >> 4) << 16) |
         ((uint64_t)(sbo >> 4) << 32) | (1ull << 46);
}

__device__ __forceinline__ void umma_f16(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc,
                                         uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(d_tmem),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate));
}

// `mbar` is arrived at once every product issued before is complete
__device__ __forceinline__ void umma_commit(uint32_t mbar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(mbar)
               : "memory");
}

}  // namespace sfm
