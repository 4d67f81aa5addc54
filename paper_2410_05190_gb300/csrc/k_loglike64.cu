// k_loglike64.cu -- double-precision likelihood: the method of Eqs. 1-3 with the marginalised
// forms of Sec. III, every bin to FP64 accuracy.  It is the double-precision GPU baseline that
// the mixed kernels are measured against, and the path of the FP64 workload.
//
// loglike_fp64_kernel (no, phase, or phase and distance marginalisation).  An FP64 instruction
// holds a quarter of an SM for 64 clocks on the GB300, so a bin that evaluates its nine-term
// phase, a sincospi and a complex multiply-add in FP64 (the version before) costs 3750 clocks
// per warp.  Every one of these quantities is bounded, and 64-bit integers carry them
// (fixed.cuh): per bin and warp
//   * the phase in turns modulo one, sum_j C_j B_j(f_k), 29 multiply-adds of 32-bit halves with
//     a unit of 2^-56 of the sample's largest phase term on the grid.  FP64 rounds each bin's own
//     terms at 2^-53: coarser where they are largest, finer where they have fallen below an
//     eighth of that;
//   * its sine and cosine to 2.7e-17 (a table of 32 entries held one per lane, fetched by
//     shuffles, and the Taylor series of the rest: 36 multiply-adds);
//   * the multiply-add with the data, scaled by the largest value of 32 bins, into 64-bit sums
//     (14 multiply-adds; exact but for 2^-56 of the products), which FP64 gathers per 32 bins.
// A warp takes 32 samples, one per lane, and 32-bin chunks of the grid: the lanes load and
// convert one bin each, and all read the converted bins back from shared memory.  A cluster of
// CTAs shares a tile of 32 samples, its warps taking the chunks in turn, and folds the sums
// through distributed shared memory in a fixed order, so the launch needs no scratch.  The
// per-sample set-up is spread over the CTA's warps, and the distance integral's nodes over the
// cluster's warps.  A sample with phase terms beyond 2^40 turns, and all samples on 32 bins with
// data that are not finite, are summed in FP64 per bin.  Bound by the integer multiply-adds (86
// per warp and bin, 4 clocks each).  Measured on a GB300, 4096 samples: 52.4 ms before and 6.6 ms
// now on 128,513 bins with phase and distance marginalised; 291 us and 56 us on 1969 bins (240
// live) with the phase marginalised.
//
// loglike_fp64_time_kernel (time marginalisation): one warp per sample, lanes over bins, every
// bin in FP64; the per-bin integrand a_k = A sum_d P_d c_dk e^(-i phi_dk) of 32
// bins at a time is staged in shared memory; lane l accumulates
// Re z_j = sum_k Re(a_k) cos(2 pi f_k tau_j) + Im(a_k) sin(2 pi f_k tau_j) for the shifts
// j = l, l + 32, ...; the warp then takes ln mean_j exp(Re z_j - H/2).
#include <cooperative_groups.h>

#include <algorithm>
#include <cmath>

#include "fixed.cuh"
#include "internal.h"
#include "marg.cuh"

namespace mbis {
namespace {

constexpr int kThreads64 = 256;
constexpr int kMaxShiftsPerLane = 8;  // up to 256 shifts

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

__device__ __forceinline__ double warp_max(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

struct Response {
  double pr[kMaxDet], pim[kMaxDet], dt[kMaxDet];
};

// sum over detectors of c_dk e^(-i (Psi_k + 2 pi f_k dt_d)) weighted by P_d (the fold table
// already carries P_d and the delays)
__device__ __forceinline__ double2 bin_term(const LikeArgs& a, const PhaseCoeffs& pc, const Response& r, int32_t k) {
  const int32_t n = a.n_bins;
  double t = pc.cst;
#pragma unroll
  for (int j = 0; j < kNumBasis; ++j) t = fma(pc.C[j], a.basis[(int64_t)j * n + k], t);
  if (a.fold) {
    double sn, cs;
    sincospi(2.0 * t, &sn, &cs);  // e^(-i Psi) = cs - i sn
    const double2 c = a.cfold64[k];
    return make_double2(c.x * cs + c.y * sn, c.y * cs - c.x * sn);
  }
  const double f = a.f_lo + (double)k * a.df;
  double zr = 0.0, zi = 0.0;
  for (int d = 0; d < a.n_det; ++d) {
    double sn, cs;
    sincospi(2.0 * fma(f, r.dt[d], t), &sn, &cs);
    const double2 c = a.cdet64[(int64_t)d * n + k];
    const double xr = c.x * cs + c.y * sn, xi = c.y * cs - c.x * sn;
    zr += r.pr[d] * xr - r.pim[d] * xi;
    zi += r.pr[d] * xi + r.pim[d] * xr;
  }
  return make_double2(zr, zi);
}

__global__ void __launch_bounds__(kThreads64) loglike_fp64_time_kernel(LikeArgs a) {
  __shared__ double2 sA[kThreads64 / 32][32];
  const int64_t s = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  if (s >= a.n) return;  // the whole warp leaves together

  double par[kNumSlots];
#pragma unroll
  for (int i = 0; i < kNumSlots; ++i) par[i] = a.pos[i] >= 0 ? a.theta[(int64_t)a.pos[i] * a.n + s] : a.fixed[i];
  if (a.marg & MBIS_MARG_PHASE) par[kPhic] = 0.0;
  if (a.marg & MBIS_MARG_DISTANCE) par[kDl] = 1.0;
  const bool valid = par[kMc] > 0.0 && par[kQ] > 0.0 && fabs(par[kChi1]) < 1.0 && fabs(par[kChi2]) < 1.0 &&
                     par[kDl] > 0.0 && isfinite(par[kTc]) && isfinite(par[kPhic]) && isfinite(par[kRa]) &&
                     isfinite(par[kDec]) && isfinite(par[kPsi]) && isfinite(par[kIota]);
  if (!valid) {
    if (lane == 0) a.out[s] = -INFINITY;
    return;
  }
  const PhaseCoeffs pc = phase_coeffs(par[kMc], par[kQ], par[kChi1], par[kChi2], par[kTc], par[kPhic]);
  const int32_t kcut = live_bins(par[kMc], par[kQ], a.f_lo, a.df, a.n_bins);
  const double A = amplitude(par[kMc], par[kDl]);
  const int32_t n = a.n_bins;

  Response r = {};
  double H = 0.0;
  if (a.fold) {
    H = A * A * a.tfold[kcut];
  } else {
    const double ci = cos(par[kIota]);
    for (int d = 0; d < a.n_det; ++d) {
      double fp, fc;
      antenna(a.det_x[d], a.det_y[d], par[kRa], par[kDec], par[kPsi], a.gmst, &fp, &fc);
      r.pr[d] = fp * 0.5 * (1.0 + ci * ci);
      r.pim[d] = -fc * ci;
      r.dt[d] = geocentre_delay(a.det_vertex[d], par[kRa], par[kDec], a.gmst);
      H += A * A * (r.pr[d] * r.pr[d] + r.pim[d] * r.pim[d]) * a.tdet[(int64_t)d * (n + 1) + kcut];
    }
  }

  {
    const int J = a.n_tshift;
    double zj[kMaxShiftsPerLane];
#pragma unroll
    for (int q = 0; q < kMaxShiftsPerLane; ++q) zj[q] = 0.0;
    for (int32_t k0 = 0; k0 < kcut; k0 += 32) {
      const int32_t k = k0 + lane;
      double2 t = make_double2(0.0, 0.0);
      if (k < kcut) {
        t = bin_term(a, pc, r, k);
        t.x *= A;
        t.y *= A;
      }
      sA[wib][lane] = t;
      __syncwarp();
      const int nk = min(32, kcut - k0);
      for (int kk = 0; kk < nk; ++kk) {
        const double2 ak = sA[wib][kk];
        const double2* tw = a.twiddle + (int64_t)(k0 + kk) * J;
#pragma unroll
        for (int q = 0; q < kMaxShiftsPerLane; ++q) {
          const int j = lane + 32 * q;
          if (j < J) {
            const double2 e = tw[j];
            zj[q] = fma(ak.x, e.x, fma(ak.y, e.y, zj[q]));
          }
        }
      }
      __syncwarp();
    }
    double m = -INFINITY;
#pragma unroll
    for (int q = 0; q < kMaxShiftsPerLane; ++q)
      if (lane + 32 * q < J) m = fmax(m, zj[q]);
    m = warp_max(m);
    double sum = 0.0;
#pragma unroll
    for (int q = 0; q < kMaxShiftsPerLane; ++q)
      if (lane + 32 * q < J) sum += exp(zj[q] - m);
    sum = warp_sum(sum);
    if (lane == 0) a.out[s] = m + log(sum / J) - 0.5 * H;
  }
}

// ---- no time marginalisation -------------------------------------------------------------
constexpr int kTile64 = 32;                  // samples per cluster, one per lane
constexpr int kWarps64 = kThreads64 / 32;
constexpr int kMaxCluster64 = 8;
constexpr int kPhaseInts = 20;               // 9 pairs and a pad: rows of 16-byte vectors
constexpr int kMaxTurnsExp = 40;             // phase terms below 2^40 turns

struct Fp64Args {
  LikeArgs a;
  int32_t eb[kNumBasis];  // |B_j(f_k)| < 2^eb_j on the grid
  int32_t chunk;          // bins of a chunk: 32, or 16 or 8 on grids with few chunks per warp
  double s_lo, s_hi;      // ln 1/dmax, ln 1/dmin
};

template <int ROWS>
struct Smem64 {
  static constexpr int kRow = kPhaseInts + 4 * ROWS;  // ints of one staged bin
  __align__(16) int32_t stage[kWarps64][32][kRow];
  double C[kNumBasis + 1][kTile64];                   // phase coefficients and the constant
  double pn[6][kTile64], mass[4][kTile64], amp[kTile64];
  double resp[3][ROWS][kTile64];                      // Re P, Im P, delay of each detector
  double part[kWarps64][2 * ROWS][kTile64];           // per-warp sums
  double cta[2 * ROWS][kTile64];                      // the CTA's sums
  double win[4][kTile64];                             // distance window: wlo, whi, Z, H
  double lse[2][kWarps64][kTile64], lse_cta[2][kTile64];
  int32_t win_flags[kTile64], kcut[kTile64];
};

// y - (y^n - x) / (n y^(n-1)) twice from an FP32 seed, with an FP32 reciprocal of the
// derivative: the seed's 1e-7 squares to 3e-14, whose step is exact to rounding
__device__ __forceinline__ double fifth_root(double x5, float seed) {
  double y = (double)seed;
  double y2 = y * y, y4 = y2 * y2;
  const double d = 0.2 * (double)__frcp_rn((float)y4);
  y = fma(-fma(y4, y, -x5), d, y);
  y2 = y * y;
  y4 = y2 * y2;
  return fma(-fma(y4, y, -x5), d, y);
}
__device__ __forceinline__ double cube_root(double x, float seed) {
  double y = (double)seed;
  double y2 = y * y;
  const double d = (1.0 / 3.0) * (double)__frcp_rn((float)y2);
  y = fma(-fma(y2, y, -x), d, y);
  y2 = y * y;
  return fma(-fma(y2, y, -x), d, y);
}
__device__ __forceinline__ double sixth_root(double x, float seed) {
  double y = (double)seed;
  double y2 = y * y, y5 = y2 * y2 * y;
  const double d = (1.0 / 6.0) * (double)__frcp_rn((float)y5);
  y = fma(-fma(y5, y, -x), d, y);
  y2 = y * y;
  y5 = y2 * y2 * y;
  return fma(-fma(y5, y, -x), d, y);
}

// u^(3/5) and x^(5/6) in the FP32 range of their seeds' arguments; the library's elsewhere
__device__ __forceinline__ double pow_3_5(double u) {
  if (!(u < 1e10)) return pow(u, 0.6);
  return fifth_root(u * u * u, powf((float)u, 0.6f));
}
__device__ __forceinline__ double cbrt_fast(double a) {
  if (!(a > 1e-18 && a < 1e18)) return cbrt(a);
  return cube_root(a, cbrtf((float)a));
}
__device__ __forceinline__ double pow_5_6(double x) {
  if (!(x > 1e-7 && x < 1e7)) return pow(x, 5.0 / 6.0);
  const double x2 = x * x;
  return sixth_root(x2 * x2 * x, powf((float)x, 5.0f / 6.0f));
}
__device__ __forceinline__ double rcp_any(double x) {
  return x > 1e-30 && x < 1e30 ? rcp_refined(x) : 1.0 / x;
}

// |x + i y|; the library's scaling only where a square would leave the range
__device__ __forceinline__ double modulus(double x, double y) {
  const double m2 = fma(x, x, y * y);
  return m2 > 1e-200 && m2 < 1e200 ? sqrt(m2) : hypot(x, y);
}

// the distance integrand's logarithm
__device__ __forceinline__ double dist_g(double s, double Z, double H, double c0) {
  const double u = exp(s);
  return c0 - 3.0 * s + log_i0(Z * u) - 0.5 * H * u * u;
}

template <int ROWS, bool FOLD>
__global__ void __launch_bounds__(kThreads64, ROWS == 1 ? 3 : 2) loglike_fp64_kernel(Fp64Args g) {
  namespace cg = cooperative_groups;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  Smem64<ROWS>& sm = *reinterpret_cast<Smem64<ROWS>*>(smem_raw);
  cg::cluster_group cluster = cg::this_cluster();
  const LikeArgs& a = g.a;
  const int R = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t s = (int64_t)(blockIdx.x / R) * kTile64 + lane;
  const bool active = s < a.n;
  const int32_t n = a.n_bins;

  double par[kNumSlots];
#pragma unroll
  for (int i = 0; i < kNumSlots; ++i)
    par[i] = active && a.pos[i] >= 0 ? a.theta[(int64_t)a.pos[i] * a.n + s] : a.fixed[i];
  if (a.marg & MBIS_MARG_PHASE) par[kPhic] = 0.0;
  if (a.marg & MBIS_MARG_DISTANCE) par[kDl] = 1.0;
  const bool valid = active && par[kMc] > 0.0 && par[kQ] > 0.0 && fabs(par[kChi1]) < 1.0 && fabs(par[kChi2]) < 1.0 &&
                     par[kDl] > 0.0 && isfinite(par[kTc]) && isfinite(par[kPhic]) && isfinite(par[kRa]) &&
                     isfinite(par[kDec]) && isfinite(par[kPsi]) && isfinite(par[kIota]);

  // ---- per-sample set-up, its independent parts on different warps
  if (!valid) {  // any coefficients: the sample has no live bin
    par[kMc] = par[kQ] = par[kDl] = 1.0;
    par[kChi1] = par[kChi2] = par[kTc] = par[kPhic] = par[kRa] = par[kDec] = par[kPsi] = par[kIota] = 0.0;
  }
  if (warp == 0) {
    // M = Mc T_sun u^(3/5), u = (1 + q)^2 / q = 1 / eta; a = pi M
    const double u = par[kQ] + 2.0 + rcp_any(par[kQ]);
    const double am = kPi * kTsun * par[kMc] * pow_3_5(u);
    const double inv_a = rcp_any(am);
    sm.mass[0][lane] = u;
    sm.mass[1][lane] = inv_a;
    sm.mass[2][lane] = log(am);
    sm.mass[3][lane] = cbrt_fast(am);
    // grid points strictly below the ISCO: an FP32 estimate, then exact FP64 steps
    const double fi = inv_a * (1.0 / 14.696938456699067);
    const float kf = ceilf((float)(fi - a.f_lo) * __frcp_rn((float)a.df));
    int32_t k = !(kf > 0.0f) ? 0 : (kf >= (float)n ? n : (int32_t)kf);
    while (k > 0 && a.f_lo + (double)(k - 1) * a.df >= fi) --k;
    while (k < n && a.f_lo + (double)k * a.df < fi) ++k;
    sm.kcut[lane] = valid ? k : 0;
  } else if (warp == 1) {
    const double w = rcp_any(1.0 + par[kQ]);
    const PNTerms t = pn_terms(par[kQ] * w * w, (par[kQ] - 1.0) * w, 0.5 * (par[kChi1] + par[kChi2]),
                               0.5 * (par[kChi1] - par[kChi2]));
    sm.pn[0][lane] = t.phi2;
    sm.pn[1][lane] = t.phi3;
    sm.pn[2][lane] = t.phi4;
    sm.pn[3][lane] = t.c5;
    sm.pn[4][lane] = t.a6;
    sm.pn[5][lane] = t.phi7;
  } else if (warp == 2) {
    sm.amp[lane] = 0.45643546458763845 * 0.46619407703541166 * pow_5_6(par[kMc] * kTsun) *
                   rcp_any(par[kDl] * kMpcSeconds);
  } else if (!FOLD && warp >= 4 && warp - 4 < ROWS) {
    const int d = warp - 4;
    double sp, cp, sd, cd, ss, cs;
    sincos(par[kRa] - a.gmst, &sp, &cp);
    sincos(par[kDec], &sd, &cd);
    sincos(par[kPsi], &ss, &cs);
    const double ci = cos(par[kIota]);
    double fp, fc;
    antenna_trig(a.det_x[d], a.det_y[d], sp, cp, sd, cd, ss, cs, &fp, &fc);
    sm.resp[0][d][lane] = fp * 0.5 * (1.0 + ci * ci);
    sm.resp[1][d][lane] = -fc * ci;
    sm.resp[2][d][lane] = delay_trig(a.det_vertex[d], sp, cp, sd, cd);
  }
  __syncthreads();
  if (warp < 2) {
    const double u = sm.mass[0][lane], inv_a = sm.mass[1][lane], la = sm.mass[2][lane], a13 = sm.mass[3][lane];
    const double pre = (3.0 / (256.0 * kPi)) * u;  // 3 / (128 eta) / (2 pi), turns
    if (warp == 0) {
      const double pa = pre * inv_a;
      sm.C[0][lane] = pa * inv_a * a13;                             // a^(-5/3)
      sm.C[1][lane] = pa * sm.pn[0][lane];                          // a^(-1)
      sm.C[2][lane] = pa * sm.pn[1][lane] * a13;                    // a^(-2/3)
      sm.C[3][lane] = pa * sm.pn[2][lane] * (a13 * a13);            // a^(-1/3)
      sm.C[8][lane] = par[kTc];
    } else {
      sm.C[4][lane] = pre * sm.pn[3][lane];
      sm.C[5][lane] = pre * a13 * (sm.pn[4][lane] - 6848.0 / 63.0 * la);
      sm.C[6][lane] = -pre * a13 * (6848.0 / 63.0);
      sm.C[7][lane] = pre * sm.pn[5][lane] * (a13 * a13);
      sm.C[kNumBasis][lane] = par[kPhic] * (-1.0 / kTwoPi) - 0.125 + pre * sm.pn[3][lane] * (1.0 + la);
    }
  }
  __syncthreads();

  // ---- the sample's coefficients in fixed point: every term below 2^T turns, unit 2^(T-56)
  int32_t T = 0;
#pragma unroll
  for (int j = 0; j < kNumBasis; ++j) T = max(T, exponent_above(sm.C[j][lane]) + g.eb[j]);
  T = max(T, exponent_above(sm.C[kNumBasis][lane]));
  if constexpr (!FOLD) {
#pragma unroll
    for (int d = 0; d < ROWS; ++d) T = max(T, exponent_above(sm.resp[2][d][lane]) + g.eb[kNumBasis - 1]);
  }
  const bool far = T > kMaxTurnsExp;  // this lane's bins in FP64; its neighbours' are not touched
  T = min(T, kMaxTurnsExp);
  Pair32 c[kNumBasis], cd[FOLD ? 1 : ROWS];
#pragma unroll
  for (int j = 0; j < kNumBasis; ++j) c[j] = pair32(far ? 0 : to_fixed(sm.C[j][lane], 60 - T + g.eb[j]));
  const int64_t cst = far ? 0 : to_fixed(sm.C[kNumBasis][lane], 56 - T);
  if constexpr (!FOLD) {
#pragma unroll
    for (int d = 0; d < ROWS; ++d)
      cd[d] = pair32(far ? 0 : to_fixed(sm.resp[2][d][lane], 60 - T + g.eb[kNumBasis - 1]));
  }
  const int32_t shift = T + 8;  // to 2^-64 turns
  const int32_t kcut = sm.kcut[lane];
  const int32_t kfix = far ? 0 : kcut;  // bins to sum in fixed point
  const int32_t kmax = __reduce_max_sync(0xffffffffu, kcut);
  const Pair32 trig_c = pair32(kTrigTable[lane][0]), trig_s = pair32(kTrigTable[lane][1]);

  // ---- sweep over the grid in chunks of 32 bins (or fewer)
  double zr[ROWS], zi[ROWS];
#pragma unroll
  for (int d = 0; d < ROWS; ++d) zr[d] = zi[d] = 0.0;
  const int32_t stride = g.chunk * kWarps64 * R;
  for (int32_t k0 = g.chunk * (rank * kWarps64 + warp); k0 < kmax; k0 += stride) {
    double nb[kNumBasis];
    double2 nw[ROWS];
    {
      const int32_t k = k0 + lane;
      const bool on = lane < g.chunk && k < n;
#pragma unroll
      for (int j = 0; j < kNumBasis; ++j) nb[j] = on ? __ldg(a.basis + (int64_t)j * n + k) : 0.0;
#pragma unroll
      for (int d = 0; d < ROWS; ++d) {
        const double2* w = FOLD ? a.cfold64 : a.cdet64 + (int64_t)d * n;
        nw[d] = on ? __ldg(w + k) : make_double2(0.0, 0.0);
      }
    }
    // each lane converts its bin: the basis in unit 2^(eb - 60), the data in 2^(E - 58)
    int32_t E = -1022;
#pragma unroll
    for (int d = 0; d < ROWS; ++d) E = max(E, max(exponent_above(nw[d].x), exponent_above(nw[d].y)));
    E = __reduce_max_sync(0xffffffffu, E);
    const bool slow = E > 900 || (E < -900 && E > -1022);  // the chunk's data: warp-uniform
    const int32_t k_end = min(k0 + g.chunk, kmax);
    if (!slow) {
      int32_t* row = sm.stage[warp][lane];
      int32_t v[Smem64<ROWS>::kRow];
#pragma unroll
      for (int j = 0; j < kNumBasis; ++j) {
        const Pair32 b = pair32(to_fixed(nb[j], 60 - g.eb[j]));
        v[2 * j] = b.h;
        v[2 * j + 1] = b.l;
      }
      v[18] = v[19] = 0;
#pragma unroll
      for (int d = 0; d < ROWS; ++d) {
        const Pair32 wr = pair32(to_fixed(nw[d].x, 58 - E)), wi = pair32(to_fixed(nw[d].y, 58 - E));
        v[kPhaseInts + 4 * d] = wr.h;
        v[kPhaseInts + 4 * d + 1] = wr.l;
        v[kPhaseInts + 4 * d + 2] = wi.h;
        v[kPhaseInts + 4 * d + 3] = wi.l;
      }
#pragma unroll
      for (int q = 0; q < Smem64<ROWS>::kRow / 4; ++q)
        reinterpret_cast<int4*>(row)[q] = make_int4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
    }
    __syncwarp();
    if (!slow) {
      int64_t ar[ROWS], ai[ROWS];  // unit 2^(E - 56)
#pragma unroll
      for (int d = 0; d < ROWS; ++d) ar[d] = ai[d] = 0;
#pragma unroll 1
      for (int32_t k = k0; k < k_end; ++k) {
        const int4* row = reinterpret_cast<const int4*>(sm.stage[warp][k - k0]);
        int32_t b[kPhaseInts];
#pragma unroll
        for (int q = 0; q < kPhaseInts / 4; ++q) {
          const int4 t = row[q];
          b[4 * q] = t.x;
          b[4 * q + 1] = t.y;
          b[4 * q + 2] = t.z;
          b[4 * q + 3] = t.w;
        }
        // each half's terms stay below 2^59, so ten of them fit a sum
        int64_t hi = cst, mid0 = 0, mid = 0;
#pragma unroll
        for (int j = 0; j < kNumBasis; ++j) {
          int64_t& mj = j < 5 ? mid0 : mid;
          hi = madw(c[j].h, b[2 * j], hi);
          mj = madw(c[j].h, b[2 * j + 1], mj);
          mj = madw(c[j].l, b[2 * j], mj);
        }
        hi = add_high(mid0, hi);
#pragma unroll
        for (int d = 0; d < ROWS; ++d) {
          int64_t dh = hi, dm = mid;
          if constexpr (!FOLD) {
            dh = madw(cd[d].h, b[2 * kNumBasis - 2], dh);
            dm = madw(cd[d].h, b[2 * kNumBasis - 1], dm);
            dm = madw(cd[d].l, b[2 * kNumBasis - 2], dm);
          }
          const uint64_t P = (uint64_t)add_high(dm, dh) << shift;
          const TrigCell cell = trig_cell(P);
          const Pair32 tc = {__shfl_sync(0xffffffffu, trig_c.h, cell.i), __shfl_sync(0xffffffffu, trig_c.l, cell.i)};
          const Pair32 ts = {__shfl_sync(0xffffffffu, trig_s.h, cell.i), __shfl_sync(0xffffffffu, trig_s.l, cell.i)};
          int64_t co64, si64;
          trig_eval(cell, tc, ts, co64, si64);
          const Pair32 co = pair32(co64), si = pair32(si64);
          const int4 w = row[kPhaseInts / 4 + d];  // re (h, l), im (h, l)
          if (k < kfix) add_rotated(Pair32{w.x, w.y}, Pair32{w.z, w.w}, co, si, ar[d], ai[d]);
        }
      }
      const double scale = __longlong_as_double((int64_t)(max(E, -900) - 56 + 1023) << 52);
#pragma unroll
      for (int d = 0; d < ROWS; ++d) {
        zr[d] = fma((double)ar[d], scale, zr[d]);
        zi[d] = fma((double)ai[d], scale, zi[d]);
      }
    }
    if (slow || far) {
#pragma unroll 1
      for (int32_t k = k0; k < min(k_end, kcut); ++k) {
        double t = sm.C[kNumBasis][lane];
        for (int j = 0; j < kNumBasis; ++j) t = fma(sm.C[j][lane], a.basis[(int64_t)j * n + k], t);
        for (int d = 0; d < ROWS; ++d) {
          const double td = FOLD ? t : fma(a.f_lo + (double)k * a.df, sm.resp[2][d][lane], t);
          double sn, cs;
          sincospi(2.0 * td, &sn, &cs);
          const double2 w = FOLD ? a.cfold64[k] : a.cdet64[(int64_t)d * n + k];
          zr[d] += w.x * cs + w.y * sn;
          zi[d] += w.y * cs - w.x * sn;
        }
      }
    }
    __syncwarp();
  }
#pragma unroll
  for (int d = 0; d < ROWS; ++d) {
    sm.part[warp][2 * d][lane] = zr[d];
    sm.part[warp][2 * d + 1][lane] = zi[d];
  }
  __syncthreads();
  for (int q = warp; q < 2 * ROWS; q += kWarps64) {
    double v = sm.part[0][q][lane];
#pragma unroll
    for (int w = 1; w < kWarps64; ++w) v += sm.part[w][q][lane];
    sm.cta[q][lane] = v;
  }
  cluster.sync();
  const bool dist = a.marg == (MBIS_MARG_PHASE | MBIS_MARG_DISTANCE);
  // the cluster's sums, in rank order (every CTA needs them for its share of the distance
  // nodes, otherwise only the first)
  if (rank == 0 || dist) {
    for (int q = warp; q < 2 * ROWS; q += kWarps64) {
      double v = 0.0;
      for (int r = 0; r < R; ++r) v += cluster.map_shared_rank(&sm.cta[0][0], r)[q * kTile64 + lane];
      sm.part[0][q][lane] = v;
    }
    __syncthreads();
    if (warp == 0) {
      const double A = sm.amp[lane];
      double X = 0.0, Y = 0.0, H = 0.0;
      if constexpr (FOLD) {
        X = A * sm.part[0][0][lane];
        Y = A * sm.part[0][1][lane];
        H = A * A * a.tfold[kcut];
      } else {
#pragma unroll
        for (int d = 0; d < ROWS; ++d) {
          const double pr = sm.resp[0][d][lane], pi = sm.resp[1][d][lane];
          const double xr = sm.part[0][2 * d][lane], xi = sm.part[0][2 * d + 1][lane];
          X += pr * xr - pi * xi;
          Y += pr * xi + pi * xr;
          H += A * A * (pr * pr + pi * pi) * a.tdet[(int64_t)d * (n + 1) + kcut];
        }
        X *= A;
        Y *= A;
      }
      if (!dist) {
        double ll;
        if (a.marg == 0)
          ll = X - 0.5 * H;
        else
          ll = log_i0(modulus(X, Y)) - 0.5 * H;
        if (active) a.out[s] = valid ? ll : -INFINITY;
      } else {
        // the peak's window (marg.cuh), and which of the ranges beside it count: G has
        // at most one maximum, so a range without it is largest at its ends; one whose ends
        // lie 50 below the window's peak adds less than e^-49 (FP64 resolves e^-36)
        const double Z = modulus(X, Y);
        double wlo = g.s_lo, whi = g.s_hi;
        int32_t flags = 0;
        if (H > 0.0 && Z * Z > 14.0 * H) {
          const double u = (Z + sqrt(Z * Z - 14.0 * H)) / (2.0 * H);
          const double sig = 1.0 / sqrt(fmax(Z * u - 7.0, 1e-300));
          const double sc = log(u);
          wlo = fmax(g.s_lo, sc - 12.0 * sig);
          whi = fmin(g.s_hi, sc + 12.0 * sig);
          if (wlo < whi) {
            const float Zf = (float)Z, Hf = (float)H;
            const double sp = fmin(fmax(sc, g.s_lo), g.s_hi);
            const float up = expf((float)sp), phi = log_i0_minus_x_f(Zf * up);
            auto below = [&](double at) { return dist_node_g((float)(at - sp), Zf, Hf, up, phi) < -50.0f; };
            flags = 1 | (wlo > g.s_lo && !(below(g.s_lo) && below(wlo)) ? 2 : 0) |
                    (whi < g.s_hi && !below(whi) ? 4 : 0);
          }
        }
        sm.win[0][lane] = wlo;
        sm.win[1][lane] = whi;
        sm.win[2][lane] = Z;
        sm.win[3][lane] = H;
        sm.win_flags[lane] = flags;
      }
    }
  }
  if (dist) {
    // the nodes of the rules, shared by the cluster's warps
    __syncthreads();
    const double wlo = sm.win[0][lane], whi = sm.win[1][lane], Z = sm.win[2][lane], H = sm.win[3][lane];
    const int32_t flags = sm.win_flags[lane];
    const double* x48 = a.gl;
    const double* w48 = a.gl + kGL48;
    const double* x8 = a.gl + 2 * kGL48;
    const double* w8 = a.gl + 2 * kGL48 + kGL8;
    const double c0 = a.dist.c0;
    LogSumExp L;
    for (int i = rank * kWarps64 + warp; i < kGL48 + 18 * kGL8 + kGL48; i += kWarps64 * R) {
      // node i: the window's 48, then 8 panels of 8 to its left and right; without a window
      // 24 panels of 8 over the whole range
      double lo = g.s_lo, hi = g.s_hi, x = 0.0, w = 0.0;
      int panel = 0, panels = 24;
      bool on = valid;
      if (flags & 1) {
        if (i < kGL48) {
          lo = wlo;
          hi = whi;
          panels = 1;
          x = x48[i];
          w = w48[i];
        } else {
          const int q = i - kGL48;  // 0..63 left, 64..127 right
          const bool right = q >= 64;
          on = on && q < 128 && (flags & (right ? 4 : 2));
          lo = right ? whi : g.s_lo;
          hi = right ? g.s_hi : wlo;
          panels = 8;
          panel = (q & 63) / kGL8;
          x = x8[q % kGL8];
          w = w8[q % kGL8];
        }
      } else {
        panel = i / kGL8;
        on = on && panel < 24;
        x = x8[i % kGL8];
        w = w8[i % kGL8];
      }
      if (on) {
        const double h = (hi - lo) / panels, mid = lo + (panel + 0.5) * h, half = 0.5 * h;
        L.add(dist_g(mid + half * x, Z, H, c0), half * w);
      }
    }
    sm.lse[0][warp][lane] = L.m;
    sm.lse[1][warp][lane] = L.acc;
    __syncthreads();
    if (warp == 0) {
      LogSumExp S;
      for (int w = 0; w < kWarps64; ++w)
        if (!(sm.lse[1][w][lane] == 0.0)) S.add(sm.lse[0][w][lane], sm.lse[1][w][lane]);
      sm.lse_cta[0][lane] = S.m;
      sm.lse_cta[1][lane] = S.acc;
    }
    cluster.sync();
    if (rank == 0 && warp == 0) {
      LogSumExp S;
      for (int r = 0; r < R; ++r) {
        const double* o = cluster.map_shared_rank(&sm.lse_cta[0][0], r);
        if (!(o[kTile64 + lane] == 0.0)) S.add(o[lane], o[kTile64 + lane]);
      }
      if (active) a.out[s] = valid ? S.value() : -INFINITY;
    }
  }
  cluster.sync();  // a CTA's shared memory outlives the other CTAs' reads
}

template <int ROWS, bool FOLD>
cudaError_t launch_fp64(const Fp64Args& g, int R, int64_t tiles, cudaStream_t s) {
  auto kernel = loglike_fp64_kernel<ROWS, FOLD>;
  constexpr int kBytes = (int)sizeof(Smem64<ROWS>);
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kBytes);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(tiles * R));
  cfg.blockDim = dim3(kThreads64);
  cfg.dynamicSmemBytes = kBytes;
  cfg.stream = s;
  cudaLaunchAttribute attr = {};
  attr.id = cudaLaunchAttributeClusterDimension;
  attr.val.clusterDim.x = (unsigned)R;
  attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  e = cudaLaunchKernelEx(&cfg, kernel, g);
  const cudaError_t sticky = cudaGetLastError();
  return e != cudaSuccess ? e : sticky;
}

// smallest e with |x| < 2^e
int32_t exponent_bound(double x) { return x == 0.0 ? 0 : std::ilogb(std::fabs(x)) + 1; }

}  // namespace

cudaError_t launch_loglike_fp64(const LikeArgs& a, cudaStream_t s) {
  if (a.n <= 0) return cudaSuccess;
  if (a.marg == MBIS_MARG_TIME) {
    const int64_t blocks = (a.n * 32 + kThreads64 - 1) / kThreads64;
    loglike_fp64_time_kernel<<<(unsigned)blocks, kThreads64, 0, s>>>(a);
    return cudaGetLastError();
  }
  Fp64Args g;
  g.a = a;
  // bounds of the basis on the grid: each function is monotonic but f^(1/3) ln f, whose one
  // extremum, -3/e at f = e^-3, is below 2 in magnitude
  const double f_hi = a.f_lo + a.df * (double)(a.n_bins - 1);
  for (int j = 0; j < kNumBasis; ++j)
    g.eb[j] = std::max(exponent_bound(basis(j, a.f_lo)), exponent_bound(basis(j, f_hi)));
  g.eb[6] = std::max(g.eb[6], 1);
  g.s_lo = -std::log(a.dmax);
  g.s_hi = -std::log(a.dmin);
  const int64_t tiles = (a.n + kTile64 - 1) / kTile64;
  // CTAs per tile: enough for four waves of the SMs, and on long grids so many that a warp
  // sweeps at most 1024 bins (the last wave then idles little); but at least a 32-bin chunk for
  // every warp.  At most eight: clusters of sixteen leave more of a GPC's CTA slots empty (4096
  // samples of 128,513 bins: 8.06 ms at 16, 6.86 at 8, 6.96 at 4).
  int R = 1;
  while (R < kMaxCluster64 && (int64_t)kThreads64 * 2 * R <= a.n_bins &&
         (tiles * R < 608 || a.n_bins > 1024 * kWarps64 * R))
    R *= 2;
  // a signal often ends well inside the grid: with under sixteen chunks of 32 bins per warp,
  // narrower chunks keep all warps at work on its live bins
  g.chunk = 32;
  while (g.chunk > 8 && a.n_bins < 16 * g.chunk * kWarps64 * R) g.chunk /= 2;
  if (a.fold) return launch_fp64<1, true>(g, R, tiles, s);
  switch (a.n_det) {
    case 1: return launch_fp64<1, false>(g, R, tiles, s);
    case 2: return launch_fp64<2, false>(g, R, tiles, s);
    case 3: return launch_fp64<3, false>(g, R, tiles, s);
    default: return launch_fp64<4, false>(g, R, tiles, s);
  }
}

}  // namespace mbis
