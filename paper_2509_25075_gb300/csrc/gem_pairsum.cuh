// A running float32 sum that loses nothing: a pair (value, error of the value)
// by Knuth's two-sum, whose second member is itself summed by two-sum.  What
// rounding takes from that is handed back to the caller, for a wider sum.
// Plain C++ without CUDA, so that the arithmetic can be tested on the host.
#pragma once

#ifdef __CUDACC__
#define GEM_HD __host__ __device__ __forceinline__
#else
#define GEM_HD inline
#endif

namespace gem {

// a + b = s + (returned error), exactly (no overflow; round to nearest).
GEM_HD float two_sum(float a, float b, float &s) {
  s = a + b;
  const float w = s - a;
  return (a - (s - w)) + (b - w);
}

// Adds v to the pair (value, error): value + error + (returned rest) is the old
// value + error + v, exactly.  The rest is zero unless the terms of the sum
// span more than 48 bits.
GEM_HD float pair_add(float &value, float &error, float v) {
  return two_sum(error, two_sum(value, v, value), error);
}

}  // namespace gem
