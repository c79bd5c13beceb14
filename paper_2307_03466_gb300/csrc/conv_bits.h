// Bit patterns of float -> double and double -> float, in integer operations alone: on the
// FP64 pipe a conversion takes as long as two FP64 additions.  Exact, or rounded to nearest
// even, for every input, with no hardware conversion left for special values: the compiler
// predicates such a branch instead of jumping over it, and the pipe is taken all the same.
// (Check of 1M to 13M nonzeros, FP32 iterates, columns / rows: multicommodity flow
// 336 / 233 -> 262 / 161 us, packing/covering 50k x 100k 28.8 / 44.5 -> 23.5 / 34.7.)
#pragma once

#include <cstdint>

#ifdef __CUDACC__
#define SCYLLA_BITS __host__ __device__ __forceinline__
#else
#define SCYLLA_BITS inline
#endif

namespace scylla {

// b: the bits of f, or of f * 2^100 (exact) where |f| < 2^-100 (small), subnormals among
// them.  The exponent is rebiased by 1023 - 127, the mantissa shifted into place.
SCYLLA_BITS uint64_t f64_bits(uint32_t b, bool small) {
  const uint32_t a = b & 0x7fffffffu;
  uint32_t bias = small ? 796u << 20 : 896u << 20;
  if (a >= 0x7f800000u) bias = 1792u << 20;  // infinities and NaNs
  if (a == 0u) bias = 0u;
  return (uint64_t(((a >> 3) + bias) | (b & 0x80000000u)) << 32) | uint32_t(b << 29);
}

SCYLLA_BITS uint32_t f32_bits(uint64_t b) {
  const uint64_t a = b & 0x7fffffffffffffffULL;
  const int e = int(a >> 52);
  uint64_t r;
  if (e >= 897 && e <= 1150) {  // a normal number; the carry of the rounding may reach infinity
    r = a - (896ULL << 52);
    r = (r + 0x0fffffffULL + ((r >> 29) & 1ULL)) >> 29;
  } else if (e > 1150) {
    r = a > 0x7ff0000000000000ULL ? 0x7fffffffULL : 0x7f800000ULL;
  } else {  // in units of 2^-149
    const int sh = 926 - e;
    const uint64_t m = (a & 0x000fffffffffffffULL) | 0x0010000000000000ULL;
    r = sh > 53 ? 0ULL : (m + ((1ULL << (sh - 1)) - 1ULL) + ((m >> sh) & 1ULL)) >> sh;
  }
  return uint32_t(r) | (uint32_t(b >> 32) & 0x80000000u);
}

// a < b for the bits of two doubles that are not NaN; -0 counts as below +0
SCYLLA_BITS bool f64_less_bits(int64_t a, int64_t b) {
  return (a ^ ((a >> 63) & 0x7fffffffffffffffLL)) < (b ^ ((b >> 63) & 0x7fffffffffffffffLL));
}

}  // namespace scylla
