// Helpers of the tcgen05 kernels (core.cu, qrp_gram.cu).
#pragma once

#include <cstdint>

namespace tk {

constexpr unsigned long long kTcSpin = 1ull << 22;  // polls of an mbarrier before a wait gives up

// shared-memory descriptor of an operand in the no-swizzle canonical layout
__device__ __forceinline__ uint64_t umma_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
  uint64_t d = (uint64_t)((saddr & 0x3FFFFu) >> 4);
  d |= (uint64_t)((lbo >> 4) & 0x3FFFu) << 16;
  d |= (uint64_t)((sbo >> 4) & 0x3FFFu) << 32;
  d |= (uint64_t)1 << 46;  // descriptor version of this architecture; base offset 0, no swizzle
  return d;
}
// exponent e with |x| < 2^e (0 for x = 0) of a finite FP32 magnitude given by its bits
// (the exponent field, or the leading zeros of a subnormal's fraction): integer arithmetic
__device__ __forceinline__ int above_exp_f32(uint32_t b) {
  const int ef = (int)(b >> 23);
  if (ef) return ef - 126;
  return b ? -149 + 32 - __clz((int)b) : 0;
}
// bounded wait for completion `parity` of an mbarrier; false if it gave up
__device__ __forceinline__ bool tc_wait(uint32_t bar, uint32_t parity) {
  for (unsigned long long it = 0; it < kTcSpin; ++it) {
    uint32_t d;
    asm volatile(
        "{ .reg .pred p; mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2; selp.u32 %0, 1, 0, p; }"
        : "=r"(d)
        : "r"(bar), "r"(parity)
        : "memory");
    if (d) return true;
    if (it > 32) __nanosleep(64);
  }
  return false;
}

}  // namespace tk
