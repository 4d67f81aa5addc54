// fixed.cuh -- fixed-point helpers of the double-precision kernels (host and device).
//
// The GB300 runs an FP64 instruction in 64 clocks per warp and SM quarter, a 32 x 32 + 64-bit
// integer multiply-add in 4, a shift, an add or a logical operation in 2 (measured).  Quantities
// whose magnitude is bounded -- a phase in turns, a sine or cosine, data scaled by their largest
// value -- therefore keep FP64 accuracy and better as 64-bit integers split into two halves,
//   X = X1 2^b + X0,
// a product of which takes three multiply-adds:
//   A B = A1 B1 2^(2b) + (A1 B0 + A0 B1) 2^b + (A0 B0, dropped).
// The FP64 likelihood takes balanced halves of b = 32 bits (Pair32 below), whose middle sum needs
// no shift; draws, logarithms and exponentials take b = 28 with 0 <= X0 < 2^28 (Pair28).  "Unit
// 2^-56" below means a 64-bit integer holding the value times 2^56.
#pragma once
#include <cstdint>
#include <cstring>

#include "fixed_tables.h"
#include "physics.cuh"

namespace mbis {

struct Pair28 {
  int32_t h, l;
};

MBIS_HD Pair28 pair28(int64_t x) { return Pair28{(int32_t)(x >> 28), (int32_t)((uint32_t)x & 0x0fffffffu)}; }

// a b + c in 64 bits.  In PTX on the device: from the C++ expression the compiler made a 64 x
// 64-bit product (3.5 multiply-adds) of halves that it could see being cut from 64-bit values.
MBIS_HD int64_t madw(int32_t a, int32_t b, int64_t c) {
#ifdef __CUDA_ARCH__
  int64_t d;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(d) : "r"(a), "r"(b), "l"(c));
  return d;
#else
  return (int64_t)a * (int64_t)b + c;
#endif
}
MBIS_HD int64_t mulw(int32_t a, int32_t b) {
#ifdef __CUDA_ARCH__
  int64_t d;
  asm("mul.wide.s32 %0, %1, %2;" : "=l"(d) : "r"(a), "r"(b));
  return d;
#else
  return (int64_t)a * (int64_t)b;
#endif
}

// (high word of a b), unsigned
MBIS_HD uint32_t mulhi_u(uint32_t a, uint32_t b) {
#ifdef __CUDA_ARCH__
  return __umulhi(a, b);
#else
  return (uint32_t)(((uint64_t)a * (uint64_t)b) >> 32);
#endif
}

// a b + c with a, b in unit 2^-56 halves: unit 2^-56
MBIS_HD int64_t mul28(Pair28 a, Pair28 b, int64_t c) {
  const int64_t mid = madw(a.h, b.l, mulw(a.l, b.h));
  return madw(a.h, b.h, c + (mid >> 28));
}

MBIS_HD uint64_t double_bits(double x) {
#ifdef __CUDA_ARCH__
  return (uint64_t)__double_as_longlong(x);
#else
  uint64_t b;
  std::memcpy(&b, &x, 8);
  return b;
#endif
}

// exponent of the smallest power of two above |x| (|x| < 2^e), from the bits; 1025 for
// infinities and NaN; zeros and subnormals count as 2^-1022
MBIS_HD int32_t exponent_above(double x) { return (int32_t)((double_bits(x) >> 52) & 0x7ff) - 1022; }

// round(x 2^e) as a 64-bit integer, by shifts (no FP64 arithmetic); |x 2^e| < 2^62
MBIS_HD int64_t to_fixed(double x, int32_t e) {
  const uint64_t b = double_bits(x);
  const int32_t be = (int32_t)((b >> 52) & 0x7ff);
  const int64_t m = be == 0 ? 0 : (int64_t)((b & 0xfffffffffffffull) | 0x10000000000000ull);  // x = m 2^(be - 1075)
  const int32_t s = be - 1075 + e;
  int64_t v;
  if (s >= 0)
    v = m << (s < 10 ? s : 10);
  else
    v = s < -54 ? 0 : (m + ((int64_t)1 << (-s - 1))) >> (-s);
  return (b >> 63) ? -v : v;
}

// Balanced 32-bit halves, X = X1 2^32 + X0 with X0 signed: the halves of a 64-bit register pair
// but for one carry, and a product's middle sum enters by its high word, so that no 64-bit
// shift (two half-rate instructions) is left in the inner loops.  With A in unit 2^-a and B in
// unit 2^-b the product has unit 2^-(a + b - 64); |A1|, |B1| <= 2^30.
struct Pair32 {
  int32_t h, l;
};

MBIS_HD Pair32 pair32(int64_t x) {
  const int32_t l = (int32_t)x;
  return Pair32{(int32_t)((uint32_t)(x >> 32) + ((uint32_t)l >> 31)), l};
}

// x + (the high word of mid, signed).  As a multiply-add by 1 it would take the pipe that bounds
// the FP64 likelihood (6.86 ms against 6.61 for 4096 samples of 128,513 bins).
MBIS_HD int64_t add_high(int64_t mid, int64_t x) { return x + (int64_t)(int32_t)(mid >> 32); }

MBIS_HD int64_t mul32(Pair32 a, Pair32 b, int64_t c) {
  return add_high(madw(a.l, b.h, mulw(a.h, b.l)), madw(a.h, b.h, c));
}

// (ar, ai) += (wr + i wi) (co - i si), every factor in halves: with w in unit 2^-58 and the
// sine and cosine in unit 2^-62 the sums have unit 2^-56.  The subtracted products negate high
// halves only: a low half of -2^31 has no negative in 32 bits.
MBIS_HD void add_rotated(Pair32 wr, Pair32 wi, Pair32 co, Pair32 si, int64_t& ar, int64_t& ai) {
  const int64_t mr = madw(wi.h, si.l, madw(wi.l, si.h, madw(wr.h, co.l, mulw(wr.l, co.h))));
  const int64_t mi = madw(-wr.h, si.l, madw(wr.l, -si.h, madw(wi.h, co.l, mulw(wi.l, co.h))));
  ar = add_high(mr, madw(wi.h, si.h, madw(wr.h, co.h, ar)));
  ai = add_high(mi, madw(wr.h, -si.h, madw(wi.h, co.h, ai)));
}

// ---- sine and cosine of a phase in turns ------------------------------------------------
// The phase P counts 2^-64 turns.  Its nearest multiple of 1/128 turn is i / 128 + q / 4
// (i = 0..31, a table entry; q the quadrant), the rest r 2^-64 turns with |r| <= 2^56.  With
// eta = r 2^-56 and zeta = eta^2 the Taylor series of the rest's angle rho = 2 pi 2^-8 eta are
//   sin rho     = eta (A0 - zeta (A1 - zeta (A2 - zeta A3))),  A_m = (2 pi 2^-8)^(2m+1) / (2m+1)!
//   cos rho - 1 = -zeta (B1 - zeta (B2 - zeta B3)),            B_m = (2 pi 2^-8)^(2m) / (2m)!
// (the first terms left out are below 2^-60), evaluated in integers; the sum formulas with the
// table entry and the quadrant give the phase's sine and cosine in unit 2^-62 with an absolute
// error of 2.7e-17 at most (3.8e-18 rms over 2 10^6 phases).
struct TrigCell {
  int32_t i, q;  // table entry, quadrant
  Pair32 x;      // eta / 4, unit 2^-64
};

MBIS_HD TrigCell trig_cell(uint64_t P) {
  const uint64_t pr = P + (1ull << 56);
  TrigCell c;
  const uint32_t hi = (uint32_t)(pr >> 32), lo = (uint32_t)pr;
  c.i = (int32_t)((hi >> 25) & 31);
  c.q = (int32_t)(hi >> 30);
  const uint32_t rh = (hi & 0x01ffffffu) - 0x01000000u;  // r's high word
  c.x.l = (int32_t)(lo << 6);
  c.x.h = (int32_t)(((rh << 6) | (lo >> 26)) + ((uint32_t)c.x.l >> 31));
  return c;
}

constexpr double kRho = kTwoPi / 256.0;
constexpr double kTwo56 = 72057594037927936.0, kTwo57 = 2.0 * kTwo56, kTwo58 = 4.0 * kTwo56;
// A0 2^66, A1 2^70, B1 2^68 (their factors 4, 64 and 16 below); A2, B2 in 2^-57, A3, B3 in 2^-58
constexpr int64_t kTrigA0 = 1811004864519280711ll, kTrigA1 = 2909163668823849ll, kTrigB1 = 88897493406080486ll;
constexpr uint32_t kTrigA2 = (uint32_t)(kRho * kRho * kRho * kRho * kRho / 120.0 * kTwo57 + 0.5);
constexpr uint32_t kTrigA3 = (uint32_t)(kRho * kRho * kRho * kRho * kRho * kRho * kRho / 5040.0 * kTwo58 + 0.5);
constexpr uint32_t kTrigB2 = (uint32_t)(kRho * kRho * kRho * kRho / 24.0 * kTwo57 + 0.5);
constexpr uint32_t kTrigB3 = (uint32_t)(kRho * kRho * kRho * kRho * kRho * kRho / 720.0 * kTwo58 + 0.5);

// cosine and sine of the cell's phase from the table entry's (tc, ts): unit 2^-62
MBIS_HD void trig_eval(const TrigCell& c, Pair32 tc, Pair32 ts, int64_t& cos_out, int64_t& sin_out) {
  // zeta / 16, unit 2^-64, and zeta's leading 31 bits
  const int64_t z64 = add_high(madw(c.x.h, c.x.l, mulw(c.x.h, c.x.l)), mulw(c.x.h, c.x.h));
  const Pair32 z = pair32(z64);
  const uint32_t x = (uint32_t)((uint64_t)z64 >> 29);
  // x (unit 2^-31) times a unit 2^-57 factor: the high word has unit 2^-56
  const uint32_t ub = mulhi_u(x, kTrigB2 - mulhi_u(x, kTrigB3));
  const uint32_t sb = mulhi_u(x, kTrigA2 - mulhi_u(x, kTrigA3));
  const int64_t u = madw((int32_t)ub, 4096, -kTrigB1);        // -16 (B1 - ...)
  const int64_t s = madw((int32_t)sb, 16384, -kTrigA1);       // -64 (A1 - ...)
  const Pair32 m = pair32(mul32(z, pair32(u), 0));            // cos rho - 1, unit 2^-64
  const Pair32 n = pair32(mul32(c.x, pair32(mul32(z, pair32(s), kTrigA0)), 0));  // sin rho
  // cos = tc + tc cm - ts sn, sin = ts + ts cm + tc sn
  int64_t mc = madw(tc.h, m.l, mulw(tc.l, m.h));
  mc = madw(-ts.h, n.l, madw(-ts.l, n.h, mc));
  int64_t ms = madw(ts.h, m.l, mulw(ts.l, m.h));
  ms = madw(tc.h, n.l, madw(tc.l, n.h, ms));
  const int64_t tc64 = ((int64_t)tc.h << 32) + tc.l, ts64 = ((int64_t)ts.h << 32) + ts.l;
  const int64_t co = add_high(mc, madw(tc.h, m.h, madw(-ts.h, n.h, tc64)));
  const int64_t si = add_high(ms, madw(ts.h, m.h, madw(tc.h, n.h, ts64)));
  // the quadrant: (cos, sin) -> (-sin, cos) per quarter turn (negation to 2^-62: ~x = -x - 1)
  const bool odd = c.q & 1;
  const int64_t c0 = odd ? si : co, s0 = odd ? co : si;
  cos_out = c0 ^ -(int64_t)(((c.q + 1) >> 1) & 1);
  sin_out = s0 ^ -(int64_t)(c.q >> 1);
}

// ---- logarithm, square root and normal draws ---------------------------------------------
MBIS_HD uint64_t umadw(uint32_t a, uint32_t b, uint64_t c) {
#ifdef __CUDA_ARCH__
  uint64_t d;
  asm("mad.wide.u32 %0, %1, %2, %3;" : "=l"(d) : "r"(a), "r"(b), "l"(c));
  return d;
#else
  return (uint64_t)a * (uint64_t)b + c;
#endif
}

MBIS_HD int32_t mulhi_s(int32_t a, int32_t b) {
#ifdef __CUDA_ARCH__
  return __mulhi(a, b);
#else
  return (int32_t)(((int64_t)a * (int64_t)b) >> 32);
#endif
}

MBIS_HD int clz64(uint64_t x) {
#ifdef __CUDA_ARCH__
  return __clzll((long long)x);
#else
  return __builtin_clzll(x);
#endif
}

constexpr int64_t kLn2_52 = 3121657384082680ll, kLn2_58 = 199786072581291495ll;  // ln 2 in 2^-52, 2^-58
constexpr int32_t kLn2_62 = -405;  // the rest of the former in 2^-62
constexpr int32_t kLn2_64 = -20;  // and the rest of the latter in 2^-64

// ln f of f = m 2^-63 in [1, 2), unit 2^-62: with c the table's 8-bit reciprocal of f's
// 1/128th, y = f c - 1 is exact and below 2^-6.9, ln f = -ln c + ln(1 + y), the series summed
// to y^8 (the rest is below 2^-65).  k = 256 c and lt = -ln c 2^62 are the entry of log_cell(m).
MBIS_HD int32_t log_cell(uint64_t m) { return (int32_t)(m >> 56) & 127; }

MBIS_HD int64_t log_frac(uint64_t m, uint32_t k, int64_t lt) {
  // f c 2^69, whose 2^69 (the 1) is zero modulo 2^64
  const uint64_t m2 = m >> 2;
  const int64_t Y = (int64_t)umadw((uint32_t)m2, k, (uint64_t)((uint32_t)(m2 >> 32) * k) << 32);
  const int64_t y = Y >> 7;  // unit 2^-62
  const Pair28 yp = pair28(y);
  const int32_t y32 = yp.h >> 2;  // unit 2^-32
  int32_t t = (int32_t)(4294967296.0 / 7.0) - mulhi_s(y32, 536870912);
  t = (int32_t)(4294967296.0 / 6.0) - mulhi_s(y32, t);
  t = (int32_t)(4294967296.0 / 5.0) - mulhi_s(y32, t);
  t = (int32_t)(4294967296.0 / 4.0) - mulhi_s(y32, t);
  // a product with yp has unit 2^-62: six more bits
  const Pair28 t4 = {t >> 4, (t & 15) << 24};
  const int64_t g = (int64_t)(kTwo56 / 3.0) - (mul28(yp, t4, 0) >> 6);
  const int64_t h = ((int64_t)1 << 55) - (mul28(yp, pair28(g), 0) >> 6);
  const int64_t y2h = mul28(pair28(mul28(yp, yp, 0)), pair28(h), 0);  // unit 2^-68
  return lt + y - (y2h >> 6);
}

// sqrt(2 t) of t = T 2^-58 > 0, unit 2^-56: an FP32 reciprocal square root and two Newton
// corrections of the root
MBIS_HD int64_t sqrt_2t(int64_t T) {
  const int lz = clz64((uint64_t)T);       // >= 1
  const int sh = (lz & 1) ? lz : lz - 1;   // odd: 2 t = M 2^-(57 + sh), M in [2^62, 2^64)
  const uint64_t M = (uint64_t)T << sh;
#ifdef __CUDA_ARCH__
  const float rs = rsqrtf((float)(uint32_t)(M >> 32));
#else
  const float rs = 1.0f / std::sqrt((float)(uint32_t)(M >> 32));
#endif
  const uint32_t Y = (uint32_t)(rs * 70368744177664.0f);  // 2^62 / sqrt(M), in [2^30, 2^31]
  const int32_t Ys = (int32_t)(Y >> 1);
  // G = sqrt(M) 2^30; e = (M 2^60 - G^2) 2^-64, dG = e Y 2^-29
  uint64_t G = umadw((uint32_t)(M >> 32), Y, umadw((uint32_t)M, Y, 0) >> 32);
  auto residual = [&]() {
    const uint32_t gh = (uint32_t)(G >> 32);
    return (int64_t)((M >> 4) - umadw(gh, gh, umadw(gh, (uint32_t)G, 0) >> 31));
  };
  int64_t e = residual();
  G += (uint64_t)((mulw((int32_t)(e >> 16), Ys) >> 12) + (mulw((int32_t)(e & 0xffff), Ys) >> 28));
  e = residual();
  G += (uint64_t)(mulw((int32_t)e, Ys) >> 28);
  const int out = (57 + sh) / 2 - 26;  // >= 3
  return (int64_t)((G + ((uint64_t)1 << (out - 1))) >> out);
}

// -ln u of u = (2 a + 1) 2^-33, unit 2^-58: the mantissa of 2 a + 1, whose table entry the
// caller looks up, and the sum
MBIS_HD int64_t minus_log_uniform(int32_t e, int64_t frac) {
  return -((int64_t)e * kLn2_58 + ((frac + ((e * kLn2_64) >> 2) + 8) >> 4));
}
MBIS_HD uint64_t uniform_mantissa(uint32_t a, int32_t& e) {
  const uint64_t w = 2 * (uint64_t)a + 1;
  const int lz = clz64(w);
  e = 30 - lz;
  return w << lz;
}

// ln x of a positive normal x = m 2^-63 2^e, unit 2^-53, from log_frac(m)
MBIS_HD int64_t log_sum(int32_t e, int64_t frac) {
  return (int64_t)e * (2 * kLn2_52) + ((frac + e * kLn2_62 + 256) >> 9);
}
struct LogArg {
  uint64_t m;
  int32_t e;
};
MBIS_HD LogArg log_arg(double x) {
  const uint64_t b = double_bits(x);
  return LogArg{((b & 0xfffffffffffffull) | 0x10000000000000ull) << 11, (int32_t)((b >> 52) & 0x7ff) - 1023};
}

// ln(sin d / d) of 0 <= d < 1/8, unit 2^-62: with t = 64 d^2 the series
// -t (1/384 + t (1/737280 + t (1/743178240 + ...))), whose next term is below 2^-58.
MBIS_HD int64_t log_sinc(double d) {
  constexpr double kUnit = 1152921504606846976.0;  // 2^60
  const Pair28 D = pair28(to_fixed(d, 59));        // 8 d, unit 2^-56
  const int64_t T = mul28(D, D, 0);
  const uint32_t t = (uint32_t)(T >> 24);
  const Pair28 tp = pair28(T);
  uint32_t b = (uint32_t)(kUnit / (37800.0 * 16777216.0)) + mulhi_u(t, (uint32_t)(kUnit / (467775.0 * 1073741824.0)));
  b = (uint32_t)(kUnit / (2835.0 * 262144.0)) + mulhi_u(t, b);
  const int64_t c = (int64_t)(kUnit / (180.0 * 4096.0)) + mulhi_u(t, b);
  const int64_t g = (int64_t)(kUnit / (6.0 * 64.0)) + mul28(tp, pair28(c), 0);
  return -(mul28(tp, pair28(g), 0) * 4);
}

// ---- exponential ---------------------------------------------------------------------------
// e^d of -700 < d <= 0 to 0.8 ulp: d = r - N ln 2 with N from the leading bits, r in (0, 0.7)
// exactly modulo 2^64 in unit 2^-63, then j / 128 + t = r, a table entry for the first and the
// Taylor series to t^6 for the second.
constexpr uint64_t kLn2_63 = 6393154322601327830ull;

MBIS_HD int32_t exp_cell(double d, int32_t& N, uint64_t& t) {
  // |d| in unit 2^-54
  const uint64_t b = double_bits(d);
  const int32_t be = (int32_t)((b >> 52) & 0x7ff), sh = be - 1075 + 54;
  const uint64_t m = be == 0 ? 0 : (b & 0xfffffffffffffull) | 0x10000000000000ull;
  const uint64_t X = sh >= 0 ? m << (sh < 11 ? sh : 11) : (sh < -54 ? 0 : (m + ((uint64_t)1 << (-sh - 1))) >> -sh);
  // |d| / ln 2 in unit 2^-21, a unit or two low
  N = (int32_t)((mulhi_u((uint32_t)(X >> 32), 3098164009u) + 4) >> 21) + 1;
  const uint64_t r = (uint64_t)N * kLn2_63 - (X << 9);
  t = r & 0xffffffffffffffull;
  return (int32_t)(r >> 56);
}

MBIS_HD double exp_eval(int32_t N, uint64_t t, int64_t e62) {
  const uint32_t t32 = (uint32_t)(t >> 24);  // unit 2^-39
  uint32_t a = (uint32_t)(4294967296.0 / 120.0) + (mulhi_u(t32, (uint32_t)(4294967296.0 / 720.0)) >> 7);
  a = (uint32_t)(4294967296.0 / 24.0) + (mulhi_u(t32, a) >> 7);
  const uint64_t b = 1537228672809129301ull + (umadw(t32, a, 0) >> 8);  // 1/6 + t (1/24 + ...), unit 2^-63
  const Pair28 tp = pair28((int64_t)t);  // 2^7 t in unit 2^-56: products have unit 2^-63
  const int64_t c = ((int64_t)1 << 62) + mul28(tp, pair28((int64_t)(b >> 7)), 0);  // 1/2 + t b
  const int64_t p = mul28(tp, pair28(mul28(tp, pair28(c >> 7), 0) >> 7), (int64_t)t);  // e^t - 1
  const uint64_t ep = (uint64_t)mul28(pair28((int64_t)((uint64_t)e62 >> 6)), pair28(p), 0);
  uint64_t m = (uint64_t)e62 + (ep >> 1);  // e^r, unit 2^-62, in [2^62, 2^64)
  const int lz = (int)(1 - (m >> 63));
  m = (m << lz) + 1024;  // rounded to 53 bits; a carry out of the top goes to the exponent
  const uint64_t carry = m < 1024;
  const uint64_t bits = ((uint64_t)(1 - lz + 1023 - N) << 52) + (carry << 52) + ((m << 1) >> 12);
#ifdef __CUDA_ARCH__
  return __longlong_as_double((long long)bits);
#else
  double v;
  std::memcpy(&v, &bits, 8);
  return v;
#endif
}

}  // namespace mbis
