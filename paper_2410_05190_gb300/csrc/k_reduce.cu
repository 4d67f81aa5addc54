// k_reduce.cu -- importance weights (Eq. 5), Kish ESS (Eq. 6) and evidence:
//   m  = max_i lw_i,  lw_i = log L_i + log pi_i - log g_i
//   S1 = sum e^(lw_i - m), S2 = sum e^(2 (lw_i - m))   (FP64),   w_i = e^(lw_i - m) / S1
//
// One launch reads the inputs once.  Each CTA takes the maximum m_b of its own samples, sums
// e^(lw - m_b) and its square, and leaves (m_b, S1_b, S2_b); the last CTA to finish (atomic
// ticket) folds the partials about m = max m_b in a fixed order with all its threads, so the
// result does not depend on scheduling.  When weights are asked for, the first launch leaves
// e^(lw - m_b) in them and a second one scales each CTA's samples by e^(m_b - m) / S1: one
// FP64 exponential per sample in all, where the FP64 pipe (2 lanes per clock per SM) and not
// HBM bounds the pass.  Measured on a GB300 at 2^18 samples with weights (device time of the
// launches): 94 us for the three launches this replaces (max 10, sum 69, weights 15: the
// sum's last thread alone folded 608 partials one dependent add after the other) against 52
// here (40 and 12); at 2^16, 78 against 30.
#include <algorithm>

#include "internal.h"

namespace mbis {
namespace {

// samples a thread keeps in registers between the maximum and the exponentials; launches of
// more than kReduceBlocks * kReduceThreads * kKeep samples read the inputs twice
constexpr int kKeep = 8;
constexpr int kWarps = kReduceThreads / 32;

__device__ __forceinline__ double log_weight(const double* ll, const double* lp, const double* lq, int64_t i) {
  return ll[i] + lp[i] - lq[i];
}

struct OpMax {
  static __device__ __forceinline__ double of(double a, double b) { return fmax(a, b); }
};
struct OpSum {
  static __device__ __forceinline__ double of(double a, double b) { return a + b; }
};

// every thread gets the fold of the CTA's values (warp shuffles, then the warps' results)
template <typename Op>
__device__ __forceinline__ double block_fold(double v, double* sh) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = Op::of(v, __shfl_xor_sync(0xffffffffu, v, o));
  __syncthreads();  // sh is free
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
  __syncthreads();
  v = sh[0];
#pragma unroll
  for (int w = 1; w < kWarps; ++w) v = Op::of(v, sh[w]);
  return v;
}

__device__ __forceinline__ bool last_block(unsigned int* counter) {
  __shared__ bool last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) last = atomicAdd(counter, 1u) == gridDim.x - 1;
  __syncthreads();
  return last;
}

// e^(lw - m); a CTA without a weight above -inf (m = -inf) has zeros, and NaN where lw is NaN
__device__ __forceinline__ double shifted_exp(double lw, double m) {
  return m > -INFINITY ? exp(lw - m) : (lw == lw ? 0.0 : lw);
}

__global__ void __launch_bounds__(kReduceThreads) reduce_kernel(int64_t n, const double* ll, const double* lp,
                                                                const double* lq, double* w, ReduceScratch scr) {
  __shared__ double sh[kWarps];
  const int64_t stride = (int64_t)gridDim.x * kReduceThreads;
  const int64_t i0 = (int64_t)blockIdx.x * kReduceThreads + threadIdx.x;
  double v[kKeep];
  double m = -INFINITY;
#pragma unroll
  for (int r = 0; r < kKeep; ++r) {
    const int64_t i = i0 + r * stride;
    v[r] = i < n ? log_weight(ll, lp, lq, i) : -INFINITY;
  }
#pragma unroll
  for (int r = 0; r < kKeep; ++r)
    if (v[r] > m) m = v[r];
  for (int64_t i = i0 + kKeep * stride; i < n; i += stride) {
    const double lw = log_weight(ll, lp, lq, i);
    if (lw > m) m = lw;
  }
  m = block_fold<OpMax>(m, sh);
  double s1 = 0.0, s2 = 0.0;
#pragma unroll
  for (int r = 0; r < kKeep; ++r) {
    const int64_t i = i0 + r * stride;
    if (i < n) {
      const double e = shifted_exp(v[r], m);
      s1 += e;
      s2 += e * e;
      if (w) w[i] = e;
    }
  }
  for (int64_t i = i0 + kKeep * stride; i < n; i += stride) {
    const double e = shifted_exp(log_weight(ll, lp, lq, i), m);
    s1 += e;
    s2 += e * e;
    if (w) w[i] = e;
  }
  s1 = block_fold<OpSum>(s1, sh);
  s2 = block_fold<OpSum>(s2, sh);
  if (threadIdx.x == 0) {
    scr.partials[3 * blockIdx.x] = m;
    scr.partials[3 * blockIdx.x + 1] = s1;
    scr.partials[3 * blockIdx.x + 2] = s2;
  }
  if (!last_block(scr.counter)) return;
  constexpr int kPer = (kReduceBlocks + kReduceThreads - 1) / kReduceThreads;
  double pm[kPer], p1[kPer], p2[kPer];
  double mm = -INFINITY;
#pragma unroll
  for (int r = 0; r < kPer; ++r) {
    const int b = r * kReduceThreads + threadIdx.x;
    const bool on = b < (int)gridDim.x;
    pm[r] = on ? __ldcg(scr.partials + 3 * b) : -INFINITY;
    p1[r] = on ? __ldcg(scr.partials + 3 * b + 1) : 0.0;
    p2[r] = on ? __ldcg(scr.partials + 3 * b + 2) : 0.0;
    mm = fmax(mm, pm[r]);
  }
  mm = block_fold<OpMax>(mm, sh);
  double a = 0.0, b2 = 0.0;
  if (mm > -INFINITY) {  // otherwise every weight is zero, whatever is NaN
#pragma unroll
    for (int r = 0; r < kPer; ++r) {
      const double f = pm[r] == mm ? 1.0 : exp(pm[r] - mm);
      a += p1[r] * f;
      b2 += p2[r] * f * f;
    }
  }
  a = block_fold<OpSum>(a, sh);
  b2 = block_fold<OpSum>(b2, sh);
  if (threadIdx.x == 0) {
    scr.result[0] = mm;
    scr.result[1] = a;
    scr.result[2] = b2;
    scr.result[3] = (double)n;
    *scr.counter = 0u;
  }
}

// the same grid as reduce_kernel: this CTA's samples are those its maximum belongs to
__global__ void __launch_bounds__(kReduceThreads) weights_kernel(int64_t n, ReduceScratch scr, double* w) {
  const double m = scr.result[0], mb = scr.partials[3 * blockIdx.x];
  const double f = (mb == m ? 1.0 : exp(mb - m)) / scr.result[1];
  const int64_t stride = (int64_t)gridDim.x * kReduceThreads;
  for (int64_t i = (int64_t)blockIdx.x * kReduceThreads + threadIdx.x; i < n; i += stride)
    w[i] = m > -INFINITY ? w[i] * f : 0.0;
}

}  // namespace

cudaError_t launch_reduce(int64_t n, const double* loglike, const double* logp, const double* logq, double* weights,
                          const ReduceScratch& scr, cudaStream_t s) {
  // one sample per thread until every CTA slot is taken: the exponentials of a small batch
  // then spread over all SMs
  const int64_t want = (n + kReduceThreads - 1) / kReduceThreads;
  const unsigned grid = (unsigned)std::max<int64_t>(1, std::min<int64_t>(want, kReduceBlocks));
  reduce_kernel<<<grid, kReduceThreads, 0, s>>>(n, loglike, logp, logq, weights, scr);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess || weights == nullptr) return e;
  weights_kernel<<<grid, kReduceThreads, 0, s>>>(n, scr, weights);
  return cudaGetLastError();
}

}  // namespace mbis
