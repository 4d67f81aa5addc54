// fpkey.cuh -- comparisons of FP64 numbers on the integer pipe: an FP64 instruction, a
// comparison included, holds its quarter of an SM for 64 clocks on the GB300.
#pragma once
#include <cstdint>

namespace mbis {

// Orders as the numbers do, with one zero.  A NaN's key lies beyond the infinities' on its
// sign's side.
__device__ __forceinline__ long long order_key(double x) {
  const long long b = __double_as_longlong(x);
  return b >= 0 ? b : (long long)(0x8000000000000000ull - (unsigned long long)b);
}

__device__ __forceinline__ bool is_nan(double x) {
  return (unsigned long long)(__double_as_longlong(x) & 0x7fffffffffffffffll) > 0x7ff0000000000000ull;
}

}  // namespace mbis
