// fpcvt.cuh -- conversions between FP64 and FP32 and range tests of FP64 numbers on the integer
// pipe, bit for bit those of the language (host and device).
//
// On the GB300 a warp's FP64 <-> FP32 conversion, like every FP64 instruction and comparison,
// holds its SM quarter's FP64 pipe for 64 to 68 clocks; the integer forms below take 5 to 12
// instructions of 1 to 2 clocks.  They are for set-ups that the FP64 pipe bounds: the tile
// assignment's (2^20 points 104 -> 65 us, device time), the folded likelihood's (2^20 BNS
// samples 63.5 -> 62.9 ms) and relative binning's (a run to a target ESS 1.73 -> 1.68 ms).  Where
// a set-up is float-float and instruction issue binds, they cost more than they save (the
// time-marginalised kernel: 2^18 samples 587 us without them, 592 with its pairs split here, 584
// with the range tests alone).  A number outside a conversion's plain range (an FP32 subnormal,
// infinity or NaN on either side) takes the language's conversion.
#pragma once
#include <cstdint>
#include <cstring>

#ifdef __CUDACC__
#define MBIS_CVT __host__ __device__ __forceinline__
#else
#define MBIS_CVT inline
#endif

namespace mbis {

MBIS_CVT void words_of(double x, uint32_t& hi, uint32_t& lo) {
#ifdef __CUDA_ARCH__
  hi = (uint32_t)__double2hiint(x);
  lo = (uint32_t)__double2loint(x);
#else
  uint64_t b;
  std::memcpy(&b, &x, 8);
  hi = (uint32_t)(b >> 32);
  lo = (uint32_t)b;
#endif
}

MBIS_CVT double double_of(uint32_t hi, uint32_t lo) {
#ifdef __CUDA_ARCH__
  return __hiloint2double((int)hi, (int)lo);
#else
  const uint64_t b = (uint64_t)hi << 32 | lo;
  double x;
  std::memcpy(&x, &b, 8);
  return x;
#endif
}

MBIS_CVT uint32_t bits_of(float x) {
#ifdef __CUDA_ARCH__
  return __float_as_uint(x);
#else
  uint32_t b;
  std::memcpy(&b, &x, 4);
  return b;
#endif
}

MBIS_CVT float float_of(uint32_t b) {
#ifdef __CUDA_ARCH__
  return __uint_as_float(b);
#else
  float x;
  std::memcpy(&x, &b, 4);
  return x;
#endif
}

// The exponent field lies in [lo, hi].
MBIS_CVT bool exponent_in(uint32_t hi_word, uint32_t lo, uint32_t hi) {
  return ((hi_word >> 20) & 0x7ffu) - lo <= hi - lo;
}

// magnitude bits of the nearest float (ties to even) of a number in the normal FP32 range;
// rounding may carry into the exponent, up to infinity's
MBIS_CVT uint32_t round_magnitude(uint32_t hi, uint32_t lo) {
  const uint32_t t = (hi << 3 | lo >> 29) + 0x40000000u;  // exponent field less 896
  return t + (((lo << 3) | (t & 1u)) > 0x80000000u ? 1u : 0u);
}

// (float)x
MBIS_CVT float to_float(double x) {
  uint32_t hi, lo;
  words_of(x, hi, lo);
  if (exponent_in(hi, 897, 1150)) return float_of(round_magnitude(hi, lo) | (hi & 0x80000000u));
  if ((hi << 1 | lo) == 0) return float_of(hi);  // a zero
  return (float)x;
}

// (double)x
MBIS_CVT double to_double(float x) {
  const uint32_t b = bits_of(x), mag = b & 0x7fffffffu;
  if (mag - 0x00800000u < 0x7f000000u) return double_of((b & 0x80000000u) | ((mag >> 3) + 0x38000000u), b << 29);
  if (mag == 0) return double_of(b, 0);
  return (double)x;
}

// (double)k of an integer that a float holds exactly for |k| < 2^24
MBIS_CVT double to_double(int32_t k) {
  return k > -(1 << 24) && k < (1 << 24) ? to_double((float)k) : (double)k;
}

// h = (float)x, l = (float)(x - (double)h).  The difference is an integer of at most 29 bits
// (round-off of the mantissa) times a power of two that FP32 holds from |x| >= 2^-74 on, so
// that the product below is exact but for the integer's own rounding.
MBIS_CVT void split_float(double x, float& h, float& l) {
  uint32_t hi, lo;
  words_of(x, hi, lo);
  if (exponent_in(hi, 949, 1149)) {
    const uint32_t sign = hi & 0x80000000u, m = round_magnitude(hi, lo);
    h = float_of(m | sign);
    int32_t r = (int32_t)(lo & 0x1fffffffu);
    if (((m ^ (lo >> 29)) & 1u) != 0) r -= 0x20000000;  // rounded away from zero
    l = (float)(sign ? -r : r) * float_of((((hi >> 20) & 0x7ffu) - 948u) << 23);
    return;
  }
  if ((hi << 1 | lo) == 0) {
    h = float_of(hi);
    l = 0.0f;
    return;
  }
  h = (float)x;
  l = (float)(x - (double)h);
}

// x > 0, |x| < 1 and finite x; false for a NaN
MBIS_CVT bool is_positive(double x) {
  uint32_t hi, lo;
  words_of(x, hi, lo);
  return (hi | lo) != 0 && (hi < 0x7ff00000u || (hi == 0x7ff00000u && lo == 0));
}
MBIS_CVT bool is_below_exp2(double x, int e) {  // |x| < 2^e, -1022 < e < 1024
  uint32_t hi, lo;
  words_of(x, hi, lo);
  return (hi & 0x7fffffffu) < (uint32_t)(1023 + e) << 20;
}
MBIS_CVT bool is_below_one(double x) { return is_below_exp2(x, 0); }
MBIS_CVT bool is_finite(double x) {
  uint32_t hi, lo;
  words_of(x, hi, lo);
  return (hi & 0x7ff00000u) != 0x7ff00000u;
}

}  // namespace mbis
