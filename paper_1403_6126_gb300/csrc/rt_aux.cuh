// What the elementwise kernels of rt_aux.cu and rt_fields.cu share.
#pragma once

#include "rt_internal.h"

namespace rtg {

inline int grid_for(long long n, int threads) {
  static int sms = 0;
  if (sms == 0) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (sms <= 0) sms = 1;
  }
  long long want = (n + threads - 1) / threads;
  long long cap = (long long)sms * 8;
  if (want < 1) want = 1;
  return (int)(want < cap ? want : cap);
}

// Range tests on the IEEE-754 bit pattern u of a double, in integer
// arithmetic (FP64 compares run at GB300's low FP64 rate): the finite
// values are the patterns with |u| below that of +infinity; the positive
// ones are 0 < u below +infinity; the non-negative ones add -0.
constexpr unsigned long long kInfBits = 0x7FF0000000000000ull, kAbsMask = 0x7FFFFFFFFFFFFFFFull,
                             kNegZero = 0x8000000000000000ull;
__device__ __forceinline__ unsigned long long bits_of(double x) { return (unsigned long long)__double_as_longlong(x); }
__device__ __forceinline__ bool finite_bits(unsigned long long u) { return (u & kAbsMask) < kInfBits; }
__device__ __forceinline__ bool positive_bits(unsigned long long u) { return u - 1ull < kInfBits - 1ull; }
__device__ __forceinline__ bool nonneg_bits(unsigned long long u) { return u < kInfBits || u == kNegZero; }

}  // namespace rtg
