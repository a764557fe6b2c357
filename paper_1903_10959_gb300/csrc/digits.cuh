// Digit words of binary64 values (kernels_ex.cu describes the scheme).
#pragma once

#include <cstdint>

namespace chfsi {

constexpr uint64_t kZeroWord = 0x8080808080808080ull;   // eight digits 0, biased by 128

__device__ __forceinline__ int expo(double v) { return (__double2hiint(v) >> 20) & 0x7ff; }

// v as an integer of up to 62 bits under the scale s = (vector's exponent field - v's own).
__device__ __forceinline__ int64_t fixed_of(double v, int s) {
  const int hi = __double2hiint(v);
  if (!(hi & 0x7ff00000)) return 0;                 // zeros and subnormal numbers vanish
  const uint64_t m = (uint64_t)(uint32_t)((hi & 0xfffff) | 0x100000) << 32 | (uint32_t)__double2loint(v);
  const int64_t t = (int64_t)(m << 9);
  return (hi < 0 ? -t : t) >> min(s, 63);
}

// Digit word of v under the scale s.
__device__ __forceinline__ uint64_t word_of(double v, int s) { return (uint64_t)fixed_of(v, s) + kZeroWord; }

}  // namespace chfsi
