// k_draw.cu -- proposal draws (g of Eq. 5) and prior densities (pi of Eq. 5).
//
// One thread per sample.  Normals come from Philox4x32-10 (philox.cuh).  Sample i of a
// call uses counter (lo32(ctr0 + i), hi32(ctr0 + i), 2, block) and key (lo32(seed),
// hi32(seed)); each block yields two Box-Muller pairs.  Because the counter names the
// sample, a sample's value does not depend on batch boundaries, launch shape or scheduling.
//
// The FP64 pipe (64 clocks per warp instruction and SM quarter) bounded the version before:
// 850 FP64 operations per sample of eleven slots, with the slot count known at run time only
// and so the normals in local memory.  Now one instantiation per slot count keeps them in
// registers, the prior's logarithms run in 64-bit fixed point (fixed.cuh), comparisons on the
// integer pipe, and the normals come in two arithmetics:
//   * contexts of MBIS_FP64: fixed point throughout -- the Box-Muller logarithm, root, sine and
//     cosine and the Cholesky sums (a normal's error is 2.8e-17 rms and 1.2e-15 at most over
//     3 10^6 draws, against 2.4e-16 and 2.9e-15 in FP64; a logarithm of the prior is within an ulp
//     up to the poles) -- which leaves FP64 a conversion and a multiply-add per slot;
//   * contexts of MBIS_MIXED: the library's FP64 functions for normals, density and prior, whose
//     last bits these samples have always had.  The mixed likelihoods round in FP32, so a sample
//     one FP64 ulp away can round to another log L (by up to 6e-8 of its spread, seen in 2 of 50
//     batches), and a refit feeds such a difference back: with this choice a seed keeps its
//     results.  (The sum of squares takes explicit multiply-adds: an unrolled chain of sums is
//     re-associated when it is contracted.)
// Measured on a GB300 (device time): 2^18 samples of 11 slots 429 us before and 61 us fixed;
// 2^16 of 5 slots 50 us before, 12 us fixed.
#include <algorithm>
#include <cmath>

#include "fixed.cuh"
#include "fpkey.cuh"
#include "internal.h"
#include "philox.cuh"

namespace mbis {
namespace {

constexpr int kDrawThreads = 128;
constexpr double kPolar = 0.12;                    // rad (log_sinc holds below 1/8)
constexpr double kPiTail = 1.2246467991473532e-16;  // pi less its nearest FP64 number

struct DrawConsts {
  double lp_const;          // the prior's log-normalisation, all slots
  double lpc[kMaxP];        // and slot by slot
  double row_scale[kMaxP];  // 2^(E_p - 56), every element of row p of scale * L below 2^E_p
  Pair28 chol[kMaxP * (kMaxP + 1) / 2];  // those elements in that unit, row by row
  double chol64[kMaxP * (kMaxP + 1) / 2];  // and in FP64
};

struct DrawTables {
  __align__(16) int4 trig[32];   // cosine and sine halves
  __align__(16) longlong2 log[128];
};

// x modulo the period, in [0, period): the quotient's floor from FP32, exact after one step either
// way; a number nearer to an end than its rounding (the step then lands on the other) is 0
__device__ __forceinline__ double wrap_period(double x, double period) {
  const float turns = __fdividef((float)x, (float)period);
  if (fabsf(turns) < 65536.0f) {
    float k = floorf(turns);
    double y = fma(-(double)k, period, x);
    if (order_key(y) < 0 || order_key(y) >= order_key(period)) {
      k += order_key(y) < 0 ? -1.0f : 1.0f;
      y = fma(-(double)k, period, x);
      if (order_key(y) < 0 || order_key(y) >= order_key(period)) y = 0.0;
    }
    return y;
  }
  double y = x - period * floor(x / period);
  if (y < 0.0) y += period;
  if (y >= period) y -= period;
  return y;
}

// ln f of a mantissa
__device__ __forceinline__ int64_t log_mantissa(const DrawTables& tb, uint64_t m) {
  const longlong2 e = tb.log[log_cell(m)];
  return log_frac(m, (uint32_t)e.x, e.y);
}

__device__ __forceinline__ int64_t log_of(const DrawTables& tb, double x) {
  const LogArg a = log_arg(x);
  return log_sum(a.e, log_mantissa(tb, a.m));
}

// cosine and sine of a phase, unit 2^-62
__device__ __forceinline__ void trig_of(const DrawTables& tb, uint64_t P, int64_t& co, int64_t& si) {
  const TrigCell c = trig_cell(P);
  const int4 t = tb.trig[c.i];
  trig_eval(c, Pair32{t.x, t.y}, Pair32{t.z, t.w}, co, si);
}

// an angle |x| < 16 rad in turns, modulo one, unit 2^-64
__device__ __forceinline__ uint64_t angle_turns(double x) {
  constexpr long long kInv2Pi = 5871781006564002453ll;  // 2^6 / (2 pi) in unit 2^-59
  const long long X = to_fixed(x, 58);
  return ((uint64_t)__mul64hi(X, kInv2Pi) << 5) | (((uint64_t)X * (uint64_t)kInv2Pi) >> 59);
}

// two normals (unit 2^-56 halves) from two words; t = (z0^2 + z1^2) / 2 in unit 2^-58
__device__ __forceinline__ int64_t box_muller(const DrawTables& tb, uint32_t a, uint32_t b, Pair28& z0, Pair28& z1) {
  int32_t e;
  const uint64_t m = uniform_mantissa(a, e);
  const int64_t t = minus_log_uniform(e, log_mantissa(tb, m));
  const Pair28 r = pair28(sqrt_2t(t));
  int64_t co, si;
  trig_of(tb, ((uint64_t)b << 32) + 0x80000000ull, co, si);
  z0 = pair28(mul28(r, pair28(co >> 6), 0));
  z1 = pair28(mul28(r, pair28(si >> 6), 0));
  return t;
}

// (a + 1/2) 2^-32, exact
__device__ __forceinline__ double uniform64(uint32_t a) {
  const uint64_t w = 2 * (uint64_t)a + 1;
  const int lz = clz64(w);
  return __longlong_as_double(((long long)(1023 + 30 - lz) << 52) | (long long)((w << lz << 1) >> 12));
}

template <int P, bool kFixed>
__global__ void __launch_bounds__(kDrawThreads) draw_kernel(DrawArgs a, DrawConsts k) {
  __shared__ DrawTables tb;
  if (threadIdx.x < 32) {
    const Pair32 c = pair32(kTrigTable[threadIdx.x][0]), s = pair32(kTrigTable[threadIdx.x][1]);
    tb.trig[threadIdx.x] = make_int4(c.h, c.l, s.h, s.l);
  }
  static_assert(kDrawThreads == 128, "a table entry per thread");
  tb.log[threadIdx.x] = make_longlong2(kLogTable[threadIdx.x][0], kLogTable[threadIdx.x][1]);
  __syncthreads();
  const int64_t i = (int64_t)blockIdx.x * kDrawThreads + threadIdx.x;
  if (i >= a.n) return;
  const uint64_t g = (a.d_ctr0 ? *a.d_ctr0 : a.ctr0) + (uint64_t)i;
  Pair28 z[P + 1];
  double zd[P + 1];
  double half_zz = 0.0;  // sum z^2 / 2
  double lp = 0.0;       // the log prior (library arithmetic)
  {
    int64_t half_zz54 = 0;  // unit 2^-54
#pragma unroll
    for (int blk = 0; blk < (P + 3) / 4; ++blk) {
      const Philox4 w = philox4x32_10((uint32_t)g, (uint32_t)(g >> 32), 2u, (uint32_t)blk, (uint32_t)a.seed,
                                      (uint32_t)(a.seed >> 32));
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int p = 4 * blk + 2 * h;
        if (p >= P) continue;
        if constexpr (kFixed) {
          const int64_t t = box_muller(tb, w.v[2 * h], w.v[2 * h + 1], z[p], z[p + 1]);
          half_zz54 += p + 1 < P ? (t + 8) >> 4 : (mul28(z[p], z[p], 0) + 4) >> 3;
        } else {
          const double r = sqrt(-2.0 * log(uniform64(w.v[2 * h])));
          double sn, cs;
          sincospi(2.0 * uniform64(w.v[2 * h + 1]), &sn, &cs);
          zd[p] = r * cs;
          zd[p + 1] = r * sn;
        }
      }
    }
    if constexpr (kFixed) {
      half_zz = (double)half_zz54 * 0x1p-54;
    } else {
      double zz = 0.0;
#pragma unroll
      for (int p = 0; p < P; ++p) zz = __fma_rn(zd[p], zd[p], zz);
      half_zz = 0.5 * zz;
    }
  }
  double mc = 0.0, q = 0.0;
  bool inside = true;
  int64_t log_sum51 = 0, polar53 = 0;  // the prior's logarithms, units 2^-51 and 2^-53
#pragma unroll
  for (int p = 0; p < P; ++p) {
    double x = a.mean[p];
    if constexpr (kFixed) {
      int64_t hi = 0, mid = 0;
#pragma unroll
      for (int r = 0; r <= p; ++r) {
        const Pair28 c = k.chol[p * (p + 1) / 2 + r];
        hi = madw(c.h, z[r].h, hi);
        mid = madw(c.h, z[r].l, madw(c.l, z[r].h, mid));
      }
      x = fma((double)(hi + (mid >> 28)), k.row_scale[p], x);
    } else {
#pragma unroll
      for (int r = 0; r <= p; ++r) x = fma(k.chol64[p * (p + 1) / 2 + r], zd[r], x);
    }
    const int id = a.ids[p];
    if (id == kRa || id == kPhic) x = wrap_period(x, kTwoPi);
    if (id == kPsi) x = wrap_period(x, kPi);
    a.theta[(int64_t)p * a.n + i] = x;
    if (id == kRa || id == kPhic || id == kPsi) {
      if constexpr (!kFixed) lp += k.lpc[p];
      continue;
    }
    inside = inside && !is_nan(x) && order_key(x) >= order_key(a.lo[p]) && order_key(x) <= order_key(a.hi[p]);
    if (id == kMc) mc = x;
    if (id == kQ) q = x;
    if constexpr (!kFixed) {
      if (id == kDec)
        lp += log(cos(x)) + k.lpc[p];
      else if (id == kIota)
        lp += log(sin(x)) + k.lpc[p];
      else if (id == kDl)
        lp += 2.0 * log(x) + k.lpc[p];
      else
        lp += k.lpc[p];
      continue;
    }
    if (id == kDec || id == kIota) {
      // ln cos(dec), ln sin(iota).  A sine in unit 2^-62 loses its relative accuracy towards the
      // poles: within kPolar of one, ln d + ln(sin d / d) of the angle d from it
      const double y = !inside ? 1.0 : id == kDec ? fabs(x) : x, pole = id == kDec ? 0.5 * kPi : kPi;
      const bool face_on = id == kIota && order_key(y) < order_key(kPolar);
      LogArg arg;
      int64_t sinc = 0;
      if (face_on || order_key(y) > order_key(pole - kPolar)) {
        const double d = face_on ? y : (pole - y) + (id == kDec ? 0.5 * kPiTail : kPiTail);
        arg = log_arg(d);
        sinc = log_sinc(d);
        if (order_key(d) == 0) inside = false;  // at the pole: ln 0
      } else {
        int64_t co, si;
        trig_of(tb, angle_turns(y), co, si);
        const uint64_t w = (uint64_t)(id == kDec ? co : si);
        const int lz = clz64(w);
        arg = LogArg{w << lz, 1 - lz};
      }
      polar53 += log_sum(arg.e, log_mantissa(tb, arg.m) + sinc);
    }
    if (id == kDl) log_sum51 += (log_of(tb, inside ? x : 1.0) + 1) >> 1;
  }
  // |d(m1, m2)/d(Mc, q)| = Mc (1 + q)^(2/5) q^(-6/5)
  if constexpr (!kFixed) {
    if ((a.flags & MBIS_PRIOR_M1M2) && inside)
      lp += 0.4 * log(mc * mc * sqrt(mc) * (1.0 + q) / (q * q * q)) - a.log_mass_norm;
    if (a.logp) a.logp[i] = inside ? lp : -INFINITY;
    if (a.logq) a.logq[i] = a.log_q_const - half_zz;
    return;
  }
  if ((a.flags & MBIS_PRIOR_M1M2) && inside) {
    const int64_t lq = log_of(tb, q);
    log_sum51 += (log_of(tb, mc) + __mul64hi(log_of(tb, 1.0 + q), 0x6666666666666666ll) - lq -
                  __mul64hi(lq, 0x3333333333333333ll) + 2) >> 2;
  }
  if (a.logp) {
    // one sum in unit 2^-53 where it holds both (|ln cos dec + ln sin iota| < 800)
    const bool both = log_sum51 < (1ll << 58) && log_sum51 > -(1ll << 58);
    lp = fma((double)(both ? polar53 + log_sum51 * 4 : polar53), 0x1p-53, k.lp_const);
    if (!both) lp = fma((double)log_sum51, 0x1p-51, lp);
    a.logp[i] = inside ? lp : -INFINITY;
  }
  if (a.logq) a.logq[i] = a.log_q_const - half_zz;
}

template <int P>
cudaError_t launch(const DrawArgs& a, const DrawConsts& k, cudaStream_t s) {
  const unsigned grid = (unsigned)((a.n + kDrawThreads - 1) / kDrawThreads);
  if (a.fixed_point)
    draw_kernel<P, true><<<grid, kDrawThreads, 0, s>>>(a, k);
  else
    draw_kernel<P, false><<<grid, kDrawThreads, 0, s>>>(a, k);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_draw(const DrawArgs& a, cudaStream_t s) {
  if (a.n <= 0) return cudaSuccess;
  DrawConsts k = {};
  for (int p = 0; p < a.P; ++p) {
    const int id = a.ids[p];
    const double lo = a.lo[p], hi = a.hi[p];
    switch (id) {
      case kRa: case kPhic: k.lpc[p] = -log(kTwoPi); break;
      case kPsi: k.lpc[p] = -log(kPi); break;
      case kDec: k.lpc[p] = -log(sin(hi) - sin(lo)); break;
      case kIota: k.lpc[p] = -log(cos(lo) - cos(hi)); break;
      case kDl: k.lpc[p] = log(3.0) - log(hi * hi * hi - lo * lo * lo); break;
      default: k.lpc[p] = (a.flags & MBIS_PRIOR_M1M2) && (id == kMc || id == kQ) ? 0.0 : -log(hi - lo); break;
    }
    k.lp_const += k.lpc[p];
    // the row of scale * L in fixed point, in units of its largest element; a factor that is
    // not finite leaves its slot's draws not finite
    double row[kMaxP];
    int32_t E = -1022;
    for (int r = 0; r <= p; ++r) {
      row[r] = k.chol64[p * (p + 1) / 2 + r] = a.scale * a.chol[p * kMaxP + r];
      E = std::max(E, exponent_above(row[r]));
    }
    const bool ok = E <= 1024;
    k.row_scale[p] = ok ? std::ldexp(1.0, E - 56) : NAN;
    for (int r = 0; r <= p; ++r) k.chol[p * (p + 1) / 2 + r] = pair28(ok ? to_fixed(row[r], 56 - E) : 0);
  }
  if (a.flags & MBIS_PRIOR_M1M2) k.lp_const -= a.log_mass_norm;
  switch (a.P) {
    case 1: return launch<1>(a, k, s);
    case 2: return launch<2>(a, k, s);
    case 3: return launch<3>(a, k, s);
    case 4: return launch<4>(a, k, s);
    case 5: return launch<5>(a, k, s);
    case 6: return launch<6>(a, k, s);
    case 7: return launch<7>(a, k, s);
    case 8: return launch<8>(a, k, s);
    case 9: return launch<9>(a, k, s);
    case 10: return launch<10>(a, k, s);
    default: return launch<11>(a, k, s);
  }
}

}  // namespace mbis
