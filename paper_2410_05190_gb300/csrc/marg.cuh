// marg.cuh -- analytic phase and numeric distance marginalisation (Sec. III: the
// likelihood is marginalised over phase and distance with analytic / numeric formulas).
//
// Phase: a uniform phi_c turns exp(Re(e^(i phi_c) Z)) into I0(|Z|).
// Distance: with Z1, H1 the overlap and norm at d_L = 1 Mpc, Z = Z1/d and H = H1/d^2, and
//   L(d) = I0(Z1/d) exp(-H1/(2 d^2)),  p(d) = 3 d^2 / (dmax^3 - dmin^3) on [dmin, dmax].
// The integral is taken in s = ln(1/d), where the integrand
//   G(s) = ln(3/(dmax^3 - dmin^3)) - 3 s + ln I0(Z1 e^s) - H1 e^(2s) / 2
// has, for a loud match (Z1^2 > 14 H1), a peak at u = e^s solving H1 u^2 - Z1 u + 7/2 = 0
// (large-argument I1/I0 ~ 1 - 1/(2x)) of width 1/sqrt(Z1 u - 7).  A 48-point Gauss-Legendre
// rule covers +-12 widths about the peak and 8-point composite rules the rest of the
// range; without a peak inside it the whole range gets a 24-panel composite 8-point rule.  Sums
// run as an online log-sum-exp: in FP64 in the double-precision kernel (k_loglike64.cu, which
// shares the nodes among its warps), in FP32 about an FP64 reference value in
// log_distance_marginal_mixed and its pieces (the mixed-precision kernels).
#pragma once
#include "physics.cuh"

namespace mbis {

// Gauss-Legendre nodes/weights on [-1, 1]: x48, w48, x8, w8 (host fills, device reads)
constexpr int kGL48 = 48, kGL8 = 8;
// a range of the mixed-precision distance rule whose largest log-integrand lies this far below
// the window's is left out
constexpr float kDistSkip = 45.0f;
constexpr int kGLSize = 2 * kGL48 + 2 * kGL8;
// The rule without a peak inside: 24 panels of 8 points over the whole distance range, whose nodes
// do not depend on the sample.  The FP32 node table goes on with their offsets d from the
// large-distance end and with expm1(d).
constexpr int kDistFull = 24 * kGL8;
constexpr int kGLTableF = kGLSize + 2 * kDistFull;  // floats of the FP32 table

#ifdef __CUDACC__
__device__ __forceinline__ double log_i0(double x) {
  x = fabs(x);
  if (x < 700.0) return log(cyl_bessel_i0(x));
  // Hankel expansion e^x / sqrt(2 pi x) * sum_k ((2k-1)!!)^2 / (k! (8x)^k)
  const double t = 1.0 / (8.0 * x);
  const double s = 1.0 + t * (1.0 + t * (4.5 + t * (37.5 + t * 459.375)));
  return x - 0.5 * log(kTwoPi * x) + log(s);
}

struct LogSumExp {
  double m = -INFINITY, acc = 0.0;
  __device__ __forceinline__ void add(double g, double w) {
    if (g > m) {
      acc = acc * exp(m - g) + w;
      m = g;
    } else {
      acc += w * exp(g - m);
    }
  }
  __device__ __forceinline__ double value() const { return m + log(acc); }
};

// ln I0(x) - x in FP32 (x >= 0), slowly varying, so FP32 keeps its absolute accuracy.  The
// polynomial approximations of Abramowitz & Stegun 9.8.1 (x < 3.75: I0 in (x/3.75)^2) and
// 9.8.2 (x >= 3.75: x^(1/2) e^(-x) I0(x) in 3.75/x) give |error| < 5e-7 in the logarithm
// over all x >= 0, with one fast logarithm, shared by the two, and no division.
__device__ __forceinline__ float log_i0_minus_x_f(float x) {
  float v;
  if (x < 3.75f) {
    const float t = x * x * (1.0f / 14.0625f);
    const float p =
        fmaf(t, fmaf(t, fmaf(t, fmaf(t, fmaf(t, fmaf(t, 0.0045813f, 0.0360768f), 0.2659732f), 1.2067492f), 3.0899424f),
                     3.5156229f),
             1.0f);
    v = p;
  } else {
    const float t = __fdividef(3.75f, x);
    const float p = fmaf(
        t,
        fmaf(t,
             fmaf(t,
                  fmaf(t, fmaf(t, fmaf(t, fmaf(t, fmaf(t, 0.00392377f, -0.01647633f), 0.02635537f), -0.02057706f),
                               0.00916281f),
                       -0.00157565f),
                  0.00225319f),
             0.01328592f),
        0.39894228f);
    v = p * rsqrtf(x);
  }
  constexpr float kLn2F = 0.69314718055994530942f;
  const float l2 = __log2f(v);
  return x < 3.75f ? fmaf(l2, kLn2F, -x) : l2 * kLn2F;
}

// (The two changes here -- a shared logarithm and a branch-free sum -- and the table of the
// whole range's nodes took the folded likelihood of 2^16 samples of 8033 bins from 163 to 151
// us and of 2^20 of 4017 bins from 3.80 to 3.62 ms, the results bit for bit the same.)
// Both branches of the running sum are one exponential of -|g - m| and one multiply-add of
// selected operands: a warp whose lanes disagree does not take two paths.
struct LogSumExpF {
  float m = -INFINITY, acc = 0.0f;
  __device__ __forceinline__ void add(float g, float w) {
    const bool up = g > m;
    const float e = __expf(-fabsf(g - m));
    acc = fmaf(up ? acc : w, e, up ? w : acc);
    m = up ? g : m;
  }
};

// G(s) - G(s_ref) at the offset d = s - s_ref, in FP32: u - u_ref = u_ref expm1(d) keeps the
// differences small, so FP32 carries ~1e-6 relative accuracy on each weight.
__device__ __forceinline__ float dist_node_e(float d, float em1, float Z, float H, float u_ref, float phi_ref) {
  const float du = u_ref * em1;
  const float u = u_ref + du;
  return Z * du - 0.5f * H * du * (2.0f * u_ref + du) - 3.0f * d + (log_i0_minus_x_f(Z * u) - phi_ref);
}
__device__ __forceinline__ float dist_node_g(float d, float Z, float H, float u_ref, float phi_ref) {
  return dist_node_e(d, expm1f(d), Z, H, u_ref, phi_ref);
}

// Node x of panel p of a composite rule over [lo, hi] (offsets from the reference point s_ref).
__device__ __forceinline__ float dist_node_at(float lo, float hi, int panels, int p, float x) {
  const float h = (hi - lo) * (1.0f / (float)panels), half = 0.5f * h;
  return fmaf(half, x, fmaf((float)p + 0.5f, h, lo));
}

// One composite rule over [lo, hi].
__device__ __forceinline__ void dist_rule_f(LogSumExpF& L, float lo, float hi, int panels, int n, const float* x,
                                            const float* w, float Z, float H, float u_ref, float phi_ref) {
  const float h = (hi - lo) * (1.0f / (float)panels), half = 0.5f * h;
  for (int p = 0; p < panels; ++p) {
#pragma unroll 4
    for (int i = 0; i < n; ++i)
      L.add(dist_node_g(dist_node_at(lo, hi, panels, p, __ldg(x + i)), Z, H, u_ref, phi_ref), half * __ldg(w + i));
  }
}
#endif

// Per-context constants of the distance marginal: c0 = ln(3 / (dmax^3 - dmin^3)), the
// large-distance end u_lo = 1 / dmax rounded to FP32 with s_lo = ln(u_lo) taken from that
// rounded value (so that the FP32 reference points below stay consistent with their
// logarithms), and the width of the range in s.
struct DistConst {
  double c0, s_lo;
  float u_lo, span;
};

inline DistConst dist_const(double dmin, double dmax) {
  DistConst d;
  d.c0 = std::log(3.0 / (dmax * dmax * dmax - dmin * dmin * dmin));
  d.u_lo = (float)(1.0 / dmax);
  d.s_lo = std::log((double)d.u_lo);
  d.span = (float)(-std::log(dmin) - d.s_lo);
  return d;
}

#ifdef __CUDACC__
// The distance marginal (48-point window of +-12 widths about the peak, 4-panel 8-point composite
// rules outside it; 24 panels of 8 points without a peak inside the range), taken in FP32 about a
// reference point s_ref (the peak, the end of the range nearest to it, or the large-distance end):
// every node contributes G(s) - G(s_ref) from dist_rule_f, and G(s_ref)
// itself is assembled in FP64 from exact products,
//   G(s_ref) = c0 - 3 s_ref + Z u_ref + [ln I0(Z u_ref) - Z u_ref] - H u_ref^2 / 2,
// so that the few terms that grow with the signal (Z u_ref, H u_ref^2 reach 10^4) keep FP64
// accuracy while the bracket, the window and the nodes run in FP32.  The reference u_ref is
// an FP32 number and s_ref = s_lo + (its offset), consistent with ln u_ref to FP32 rounding.
struct DistWindow {
  bool window;
  float lo, hi;           // the window as offsets from the reference point
  float wlo, whi, r_ref;  // the window and the reference point as offsets from s_lo
  float Z, H, u_ref, phi_ref;
};

__device__ __forceinline__ DistWindow dist_window(double Z, double H, const DistConst& dc) {
  DistWindow d;
  d.Z = to_float(Z);
  d.H = to_float(H);
  d.window = false;
  d.wlo = 0.0f;
  d.whi = dc.span;
  d.r_ref = 0.0f;
  if (d.H > 0.0f && d.Z * d.Z > 14.0f * d.H) {
    const float u = (d.Z + sqrtf(d.Z * d.Z - 14.0f * d.H)) / (2.0f * d.H);
    const float sig = rsqrtf(fmaxf(d.Z * u - 7.0f, 1e-30f));
    const float rc = logf(u / dc.u_lo);
    d.wlo = fmaxf(0.0f, rc - 12.0f * sig);
    d.whi = fminf(dc.span, rc + 12.0f * sig);
    d.window = d.wlo < d.whi;
    d.r_ref = fminf(fmaxf(rc, 0.0f), dc.span);
    if (!d.window) {  // the peak lies beyond an end: the whole range about that end
      d.wlo = 0.0f;
      d.whi = dc.span;
    }
  }
  d.u_ref = dc.u_lo * __expf(d.r_ref);
  d.phi_ref = log_i0_minus_x_f(d.Z * d.u_ref);
  d.lo = d.wlo - d.r_ref;
  d.hi = d.whi - d.r_ref;
  return d;
}

// The main rule: 48 nodes over the window; without one the whole range's, tabled for the reference
// point at the large-distance end (lo = 0).  A peak beyond the near end puts the reference there,
// where the integrand is largest and the growing terms vanish: no main rule then, dist_finish
// evaluates the range.
__device__ __forceinline__ int dist_main_count(const DistWindow& d) {
  return d.window ? kGL48 : d.lo == 0.0f ? kDistFull : 0;
}
// node i: its offset and expm1 of it
__device__ __forceinline__ float2 dist_main_node(bool window, float lo, float hi, const float* gl, int i) {
  if (!window) return make_float2(__ldg(gl + kGLSize + i), __ldg(gl + kGLSize + kDistFull + i));
  const float d = dist_node_at(lo, hi, 1, 0, __ldg(gl + i));
  return make_float2(d, expm1f(d));
}
__device__ __forceinline__ float dist_main_weight(bool window, float lo, float hi, const float* gl, int i) {
  const float h = (hi - lo) * (window ? 1.0f : 1.0f / 24.0f);
  return 0.5f * h * __ldg(gl + (window ? kGL48 + i : 2 * kGL48 + kGL8 + i % kGL8));
}

// The whole range about the near end, for the rare source inside dmin: called, so that the kernels'
// own code is that of the other two rules.
static __device__ __noinline__ LogSumExpF dist_near_range(float lo, float hi, const float* x8, float Z, float H,
                                                          float u_ref, float phi_ref) {
  LogSumExpF L;
  dist_rule_f(L, lo, hi, 24, kGL8, x8, x8 + kGL8, Z, H, u_ref, phi_ref);
  return L;
}

// The marginal from the main rule's sum L.
__device__ __forceinline__ double dist_finish(const DistWindow& d, LogSumExpF L, double Z, double H, const DistConst& dc,
                                              const float* gl) {
  const float* x8 = gl + 2 * kGL48;
  const float* w8 = gl + 2 * kGL48 + kGL8;
  if (d.window) {
    // Outside the window: G has at most one local maximum (G' = f(x) - 3 with
    // f(x) = x I1(x)/I0(x) - (H/Z^2) x^2 rising then falling in x = Z e^s), so a range that
    // does not hold it takes its largest value at its ends.  A range whose ends lie more than
    // kDistSkip below the window's largest node is left out: its share of the integral is
    // below e^-40.  (Were the maximum inside the range, the window's nearest end would be
    // within kDistSkip of the window's largest node and the range would be summed.)
    if (d.wlo > 0.0f) {
      const float g_end = fmaxf(dist_node_g(-d.r_ref, d.Z, d.H, d.u_ref, d.phi_ref),
                                dist_node_g(d.lo, d.Z, d.H, d.u_ref, d.phi_ref));
      if (g_end > L.m - kDistSkip) dist_rule_f(L, -d.r_ref, d.lo, 4, kGL8, x8, w8, d.Z, d.H, d.u_ref, d.phi_ref);
    }
    if (d.whi < dc.span && dist_node_g(d.hi, d.Z, d.H, d.u_ref, d.phi_ref) > L.m - kDistSkip)
      dist_rule_f(L, d.hi, dc.span - d.r_ref, 4, kGL8, x8, w8, d.Z, d.H, d.u_ref, d.phi_ref);
  } else if (d.lo != 0.0f) {
    L = dist_near_range(d.lo, d.hi, x8, d.Z, d.H, d.u_ref, d.phi_ref);
  }
  const double u_ref = to_double(d.u_ref);
  const double g_ref =
      dc.c0 - 3.0 * (dc.s_lo + to_double(d.r_ref)) + Z * u_ref - 0.5 * H * u_ref * u_ref + to_double(d.phi_ref);
  return g_ref + to_double(L.m) + to_double(logf(L.acc));
}

__device__ __forceinline__ double log_distance_marginal_mixed(double Z, double H, const DistConst& dc,
                                                              const float* gl) {
  const DistWindow d = dist_window(Z, H, dc);
  LogSumExpF L;
  if (d.window) {
    dist_rule_f(L, d.lo, d.hi, 1, kGL48, gl, gl + kGL48, d.Z, d.H, d.u_ref, d.phi_ref);
  } else if (dist_main_count(d) > 0) {
#pragma unroll 4
    for (int i = 0; i < kDistFull; ++i) {
      const float2 n = dist_main_node(false, d.lo, d.hi, gl, i);
      L.add(dist_node_e(n.x, n.y, d.Z, d.H, d.u_ref, d.phi_ref), dist_main_weight(false, d.lo, d.hi, gl, i));
    }
  }
  return dist_finish(d, L, Z, H, dc, gl);
}
#endif

// host: Gauss-Legendre nodes by Newton iteration on the Legendre recurrence
inline void gauss_legendre(int n, double* x, double* w) {
  for (int i = 0; i < n; ++i) {
    double z = cos(kPi * (i + 0.75) / (n + 0.5)), dp = 0.0;
    for (int it = 0; it < 100; ++it) {
      double p0 = 1.0, p1 = z;
      for (int k = 2; k <= n; ++k) {
        const double p2 = ((2.0 * k - 1.0) * z * p1 - (k - 1.0) * p0) / k;
        p0 = p1;
        p1 = p2;
      }
      dp = n * (z * p1 - p0) / (z * z - 1.0);
      const double dz = p1 / dp;
      z -= dz;
      if (fabs(dz) < 1e-16) break;
    }
    x[i] = z;
    w[i] = 2.0 / ((1.0 - z * z) * dp * dp);
  }
}

inline void fill_gauss_legendre(double* gl) {
  gauss_legendre(kGL48, gl, gl + kGL48);
  gauss_legendre(kGL8, gl + 2 * kGL48, gl + 2 * kGL48 + kGL8);
}

// the same table rounded to FP32 (the mixed-precision marginal's copy)
inline void fill_gauss_legendre_f32(float* glf) {
  double gl[kGLSize];
  fill_gauss_legendre(gl);
  for (int i = 0; i < kGLSize; ++i) glf[i] = (float)gl[i];
}

}  // namespace mbis
