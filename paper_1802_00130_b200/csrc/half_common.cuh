// What the writers and readers of FP16 copies share (see HalfInfo in gn_kernels.h).
#pragma once
#include <cuda_runtime.h>

#include "gn_kernels.h"

namespace gn {
namespace {

constexpr int kHalfMaxExp = 120;     // |e| of a copy, and |e| + |e| of two of them, within the range of a float factor

__device__ __forceinline__ unsigned magnitude(float x) { return __float_as_uint(x) & 0x7fffffffu; }
__device__ __forceinline__ float half_scale(int e) { return __uint_as_float((unsigned)(e + 127) << 23); }     // 2^e, |e| <= 126

// e that takes magnitudes up to that of this bit pattern to [2^14, 2^15) (0 for a matrix of zeros or with an infinity or NaN)
__device__ __forceinline__ int half_exponent(unsigned amax_bits) {
  if (amax_bits == 0u || amax_bits >= 0x7f800000u) return 0;
  return max(-kHalfMaxExp, min(kHalfMaxExp, 14 - ((int)(amax_bits >> 23) - 127)));      // (denormals: as 2^-127)
}

// largest of |a|, |b|, |c| (NaN if one of them is)
__device__ __forceinline__ float max3_abs(float a, float b, float c) {
  float d;
  asm("max.NaN.abs.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}

// A sum of magnitudes that an info has in units of 2^(-e - kHalfNormExp).
constexpr int kHalfNormExp = 4;
__device__ __forceinline__ float half_norm(unsigned long long units, int e) { return (float)units * half_scale(-kHalfNormExp) * half_scale(-e); }

// Collects what decides whether a copy may be used, from the largest scaled magnitudes of runs of a row or column.
struct HalfCheck {
  unsigned low = 0xffffffffu, high = 0u;     // smallest that is not zero (less one: zeros wrap to the largest), and largest
  __device__ __forceinline__ void run(float largest) {
    const unsigned b = __float_as_uint(largest);
    low = min(low, b - 1u);
    high = max(high, b);
  }
  __device__ __forceinline__ bool low_run() const { return low < __float_as_uint(kHalfLeast) - 1u; }
  __device__ __forceinline__ bool bad() const { return low < __float_as_uint(kHalfLeast) - 1u || high > __float_as_uint(65504.f); }
};

}  // namespace
}  // namespace gn
