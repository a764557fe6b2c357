// Digit words of binary64 values (kernels_ex.cu describes the scheme).
#pragma once

#include <cstdint>

namespace chfsi {

constexpr uint64_t kZeroWord = 0x8080808080808080ull;   // eight digits 0, biased by 128

// Exponent field of v as its scale: subnormal numbers have that of the smallest
// normal ones (and no leading bit), and so have zeros.
__device__ __forceinline__ int expo(double v) { return max((__double2hiint(v) >> 20) & 0x7ff, 1); }
__device__ __forceinline__ bool nonzero(double v) { return ((__double2hiint(v) & 0x7fffffff) | __double2loint(v)) != 0; }

// v as an integer of up to 62 bits under the scale s = (vector's exponent field - v's own).
__device__ __forceinline__ int64_t fixed_of(double v, int s) {
  const int hi = __double2hiint(v);
  const uint32_t lead = min(hi & 0x7ff00000, 0x100000);
  const uint64_t m = (uint64_t)((hi & 0xfffff) | lead) << 32 | (uint32_t)__double2loint(v);
  const int64_t t = (int64_t)(m << 9);
  return (hi < 0 ? -t : t) >> min(s, 63);
}

// Digit word of v under the scale s.
__device__ __forceinline__ uint64_t word_of(double v, int s) { return (uint64_t)fixed_of(v, s) + kZeroWord; }

}  // namespace chfsi
