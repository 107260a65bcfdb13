// Shared-memory addresses, operand descriptors and bounded mbarrier waits of the
// tensor-core kernels.
#pragma once
#include <cstdint>

#include "common.cuh"

#define MM_KT 64              // K per tile: one 128-byte swizzled row of 16-bit values
#define MM_SPIN (1u << 22)    // polls after which a wait gives up

__device__ __forceinline__ unsigned mm_sa(const void* p) {
  return (unsigned)__cvta_generic_to_shared(p);
}
// shared-memory matrix descriptor: K-major, 128-byte swizzle, 8-row atoms of 1024 B
__device__ __forceinline__ uint64_t mm_desc_sw128(unsigned addr) {
  uint64_t d = 0;
  d |= (uint64_t)((addr >> 4) & 0x3FFF);
  d |= (uint64_t)1 << 16;               // leading byte offset (not used by swizzled K-major)
  d |= (uint64_t)(1024 >> 4) << 32;     // stride byte offset: 8 rows x 128 B
  d |= (uint64_t)1 << 46;               // descriptor version
  d |= (uint64_t)2 << 61;               // 128-byte swizzle
  return d;
}
__device__ __forceinline__ bool mm_wait(unsigned long long* b, unsigned parity) {
  for (unsigned it = 0; it < MM_SPIN; ++it) {
    unsigned ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(mm_sa(b)), "r"(parity)
        : "memory");
    if (ok) return true;
  }
  return false;
}
