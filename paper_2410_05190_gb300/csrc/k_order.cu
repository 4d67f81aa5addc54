// k_order.cu -- the order in which the likelihood kernels take the samples of a launch:
// most live bins first.  A CTA runs to the longest band among its samples (and a warp to the
// longest among its lanes), while a sample's result does not depend on which CTA or lanes
// it shares -- its bins past its own ISCO cut add exact zeros -- so ordering the samples by
// their live bins only removes the work a CTA would spend on its longest sample.
#include "internal.h"
#include "order.cuh"

namespace mbis {
namespace {

// The part of LikeArgs that the key needs: a kernel's parameters are copied at each launch.
struct BandKey {
  const double *mc, *q;  // null: fixed
  double mc0, q0;
  float f_lo, df, n_bins;
  int32_t gran;
  // live bins of sample i in units of gran bins (rounded up), estimated in FP32: the estimate
  // only steers the order; each CTA still runs to the exact cut of its samples
  __device__ __forceinline__ int32_t operator()(int64_t i) const {
    const float m = (float)(mc ? mc[i] : mc0), qf = (float)(q ? q[i] : q0);
    if (!(m > 0.0f) || !(qf > 0.0f)) return 0;
    const float m_sec = m * (float)kTsun * powf(1.0f + qf, 1.2f) * powf(qf, -0.6f);
    const float fi = 1.0f / (46.172139f * m_sec);  // 6^(3/2) pi M
    const float k = fminf(fmaxf(ceilf((fi - f_lo) / df), 0.0f), n_bins);
    return ((int32_t)k + gran - 1) / gran;
  }
};

// one CTA: counts -> first slot of each key, keys in decreasing order.  Every thread owns a
// contiguous run of keys, read and written as a whole; long key ranges (a bin pair per key on
// a 128k-bin grid) go through shared memory in coalesced pieces.
constexpr int kScanThreads = 1024;
constexpr int kScanPer = 8;

__global__ void __launch_bounds__(kScanThreads) order_scan_kernel(int32_t n_keys, int32_t* hist) {
  __shared__ int32_t warp_tot[32];
  __shared__ int32_t piece[kScanThreads * (kScanPer + 1)];  // padded: a thread's run is conflict-free
  __shared__ int32_t s_carry;
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  if (t == 0) s_carry = 0;
  constexpr int kPiece = kScanThreads * kScanPer;
  for (int32_t r0 = 0; r0 < n_keys; r0 += kPiece) {  // ranks r: key n_keys - 1 - r
    for (int j = t; j < kPiece; j += kScanThreads) {
      const int32_t r = r0 + j;
      piece[j + j / kScanPer] = r < n_keys ? hist[n_keys - 1 - r] : 0;
    }
    __syncthreads();
    int32_t* mine = piece + t * (kScanPer + 1);
    int32_t local = 0;
#pragma unroll
    for (int j = 0; j < kScanPer; ++j) local += mine[j];
    int32_t incl = local;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int32_t v = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += v;
    }
    if (lane == 31) warp_tot[warp] = incl;
    __syncthreads();
    if (warp == 0) {
      int32_t v = warp_tot[lane];
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int32_t u = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += u;
      }
      warp_tot[lane] = v;  // inclusive over warps
    }
    __syncthreads();
    int32_t run = s_carry + incl - local + (warp > 0 ? warp_tot[warp - 1] : 0);
#pragma unroll
    for (int j = 0; j < kScanPer; ++j) {
      const int32_t c = mine[j];
      mine[j] = run;
      run += c;
    }
    __syncthreads();
    if (t == 0) s_carry += warp_tot[31];
    for (int j = t; j < kPiece; j += kScanThreads) {
      const int32_t r = r0 + j;
      if (r < n_keys) hist[n_keys - 1 - r] = piece[j + j / kScanPer];
    }
    __syncthreads();
  }
}

}  // namespace

cudaError_t launch_order_scan(int32_t n_keys, int32_t* counts, cudaStream_t s) {
  order_scan_kernel<<<1, kScanThreads, 0, s>>>(n_keys, counts);
  return cudaGetLastError();
}

int32_t order_keys(int32_t n_bins, int32_t gran) { return (n_bins + gran - 1) / gran + 1; }

cudaError_t launch_sample_order(const LikeArgs& a, int32_t gran, int32_t* hist, int32_t* perm, cudaStream_t s) {
  BandKey key;
  key.mc = a.pos[kMc] >= 0 ? a.theta + (int64_t)a.pos[kMc] * a.n : nullptr;
  key.q = a.pos[kQ] >= 0 ? a.theta + (int64_t)a.pos[kQ] * a.n : nullptr;
  key.mc0 = a.fixed[kMc];
  key.q0 = a.fixed[kQ];
  key.f_lo = (float)a.f_lo;
  key.df = (float)a.df;
  key.n_bins = (float)a.n_bins;
  key.gran = gran;
  return launch_order(a.n, order_keys(a.n_bins, gran), key, hist, perm, s);
}

}  // namespace mbis
