// k_reduce.cu -- importance weights (Eq. 5), Kish ESS (Eq. 6) and evidence:
//   m  = max_i lw_i,  lw_i = log L_i + log pi_i - log g_i
//   S1 = sum e^(lw_i - m), S2 = sum e^(2 (lw_i - m))   (FP64),   w_i = e^(lw_i - m) / S1
//
// One launch reads the inputs once.  Each CTA takes the maximum m_b of its own samples, sums
// e^(lw - m_b) and its square, and leaves (m_b, S1_b, S2_b); the last CTA to finish (atomic
// ticket) folds the partials about m = max m_b in a fixed order with all its threads, so the
// result does not depend on scheduling.  When weights are asked for, the first launch leaves lw
// in them and a second one makes e^(lw - m) / S1 of it: e^(lw - m_b) scaled by e^(m_b - m) / S1
// would save the second exponential and carry the rounding of a further one.
// The FP64 pipe (64 clocks per warp instruction and SM quarter) bounds the pass and not HBM:
// the exponentials run in fixed point (fixed.cuh: 0.76 ulp at most, 0.31 rms, where FP64 took
// some 30 instructions), the maxima on the integer pipe, and a warp's two sums fold with five
// adds between them, which leaves five FP64 instructions per sample.  Measured on a GB300 with
// weights (device time): 94 us at 2^18 samples, 78 at 2^16 and 74 at 4096 for the three launches
// of the first version (its sum ended in one thread adding 608 partials), 29 (22 and 6), 17 and
// 14 here.
#include <algorithm>

#include "fixed.cuh"
#include "fpkey.cuh"
#include "internal.h"

namespace mbis {
namespace {

// samples a thread keeps in registers between the maximum and the exponentials; launches of
// more than kReduceBlocks * kReduceThreads * kKeep samples read the inputs twice
constexpr int kKeep = 8;
constexpr int kWarps = kReduceThreads / 32;
static_assert(kWarps == 8, "the second fold takes one lane per warp in each half of a warp");
constexpr long long kKeyMin = -0x7ff0000000000000ll;  // order_key(-inf)

__device__ __forceinline__ double log_weight(const double* ll, const double* lp, const double* lq, int64_t i) {
  return ll[i] + lp[i] - lq[i];
}

__device__ __forceinline__ double from_key(long long k) {
  return __longlong_as_double(k >= 0 ? k : (long long)(0x8000000000000000ull - (unsigned long long)k));
}

// every thread gets the largest key
__device__ __forceinline__ long long block_max(long long v, long long* sh) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = max(v, (long long)__shfl_xor_sync(0xffffffffu, v, o));
  __syncthreads();  // sh is free
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
  __syncthreads();
  v = sh[0];
#pragma unroll
  for (int w = 1; w < kWarps; ++w) v = max(v, sh[w]);
  return v;
}

// thread 0 gets both sums: the lower half of a warp folds a, the upper b
__device__ __forceinline__ void block_sum2(double& a, double& b, double* sh) {
  const int lane = threadIdx.x & 31;
  double v = (lane < 16 ? a : b) + __shfl_xor_sync(0xffffffffu, lane < 16 ? b : a, 16);
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((lane & 15) == 0) sh[(lane >> 4) * kWarps + (threadIdx.x >> 5)] = v;
  __syncthreads();
  if (threadIdx.x < 32) {
    v = (lane & 15) < kWarps ? sh[(lane >> 4) * kWarps + (lane & 15)] : 0.0;
#pragma unroll
    for (int o = kWarps / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    a = v;
    b = __shfl_sync(0xffffffffu, v, 16);
  }
}

__device__ __forceinline__ bool last_block(unsigned int* counter) {
  __shared__ bool last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) last = atomicAdd(counter, 1u) == gridDim.x - 1;
  __syncthreads();
  return last;
}

// e^(x - m) for x <= m; NaN where x is (or both are infinite); a CTA without a weight above
// -inf (m = -inf) has zeros
__device__ __forceinline__ double shifted_exp(double x, double m) {
  const double d = x - m;
  if (is_nan(d)) return is_nan(x) || order_key(m) > kKeyMin ? d : 0.0;
  const long long k = order_key(d);
  if (k < order_key(-700.0)) return k < order_key(-746.0) ? 0.0 : exp(d);
  int32_t n;
  uint64_t t;
  const int32_t j = exp_cell(d, n, t);
  return exp_eval(n, t, __ldg(reinterpret_cast<const long long*>(kExpTable) + j));
}

__global__ void __launch_bounds__(kReduceThreads) reduce_kernel(int64_t n, const double* ll, const double* lp,
                                                                const double* lq, double* w, ReduceScratch scr) {
  __shared__ long long sh_max[kWarps];
  __shared__ double sh_sum[2 * kWarps];
  const int64_t stride = (int64_t)gridDim.x * kReduceThreads;
  const int64_t i0 = (int64_t)blockIdx.x * kReduceThreads + threadIdx.x;
  double v[kKeep];
  long long top = kKeyMin;
#pragma unroll
  for (int r = 0; r < kKeep; ++r) {
    const int64_t i = i0 + r * stride;
    if (i < n) v[r] = log_weight(ll, lp, lq, i);
  }
#pragma unroll
  for (int r = 0; r < kKeep; ++r)
    if (i0 + r * stride < n && !is_nan(v[r])) top = max(top, order_key(v[r]));
  for (int64_t i = i0 + kKeep * stride; i < n; i += stride) {
    const double lw = log_weight(ll, lp, lq, i);
    if (!is_nan(lw)) top = max(top, order_key(lw));
  }
  const double m = from_key(block_max(top, sh_max));
  double s1 = 0.0, s2 = 0.0;
  auto take = [&](int64_t i, double lw) {
    const double e = shifted_exp(lw, m);
    s1 += e;
    s2 = fma(e, e, s2);
    if (w) w[i] = lw;
  };
#pragma unroll
  for (int r = 0; r < kKeep; ++r) {
    const int64_t i = i0 + r * stride;
    if (i < n) take(i, v[r]);
  }
  for (int64_t i = i0 + kKeep * stride; i < n; i += stride) take(i, log_weight(ll, lp, lq, i));
  block_sum2(s1, s2, sh_sum);
  if (threadIdx.x == 0) {
    scr.partials[3 * blockIdx.x] = m;
    scr.partials[3 * blockIdx.x + 1] = s1;
    scr.partials[3 * blockIdx.x + 2] = s2;
  }
  if (!last_block(scr.counter)) return;
  constexpr int kPer = (kReduceBlocks + kReduceThreads - 1) / kReduceThreads;
  double pm[kPer], p1[kPer], p2[kPer];
  top = kKeyMin;
#pragma unroll
  for (int r = 0; r < kPer; ++r) {
    const int b = r * kReduceThreads + threadIdx.x;
    const bool on = b < (int)gridDim.x;
    pm[r] = on ? __ldcg(scr.partials + 3 * b) : -INFINITY;
    p1[r] = on ? __ldcg(scr.partials + 3 * b + 1) : 0.0;
    p2[r] = on ? __ldcg(scr.partials + 3 * b + 2) : 0.0;
    top = max(top, order_key(pm[r]));
  }
  top = block_max(top, sh_max);
  const double mm = from_key(top);
  s1 = s2 = 0.0;
  if (top > kKeyMin) {  // otherwise every weight is zero, whatever is NaN
#pragma unroll
    for (int r = 0; r < kPer; ++r) {
      if (r * kReduceThreads + (int)threadIdx.x >= (int)gridDim.x) continue;
      const double f = order_key(pm[r]) == top ? 1.0 : shifted_exp(pm[r], mm);
      s1 = fma(p1[r], f, s1);
      s2 = fma(p2[r], f * f, s2);
    }
  }
  block_sum2(s1, s2, sh_sum);
  if (threadIdx.x == 0) {
    scr.result[0] = mm;
    scr.result[1] = s1;
    scr.result[2] = s2;
    scr.result[3] = (double)n;
    *scr.counter = 0u;
  }
}

__global__ void __launch_bounds__(kReduceThreads) weights_kernel(int64_t n, ReduceScratch scr, double* w) {
  __shared__ double sh_inv;
  if (threadIdx.x == 0) sh_inv = 1.0 / scr.result[1];
  __syncthreads();
  const double m = scr.result[0], inv = sh_inv;
  const bool any = order_key(m) > kKeyMin;
  const int64_t stride = (int64_t)gridDim.x * kReduceThreads;
  for (int64_t i = (int64_t)blockIdx.x * kReduceThreads + threadIdx.x; i < n; i += stride)
    w[i] = any ? shifted_exp(w[i], m) * inv : 0.0;
}

// ---- the ordered form, for the refits of the ESS loop
__global__ void __launch_bounds__(kReduceThreads) ordered_max_kernel(int64_t n, const double* ll, const double* lp,
                                                                     const double* lq, ReduceScratch scr) {
  __shared__ long long sh_max[kWarps];
  const int64_t stride = (int64_t)gridDim.x * kReduceThreads;
  long long top = kKeyMin;
  for (int64_t i = (int64_t)blockIdx.x * kReduceThreads + threadIdx.x; i < n; i += stride) {
    const double lw = log_weight(ll, lp, lq, i);
    if (!is_nan(lw)) top = max(top, order_key(lw));
  }
  top = block_max(top, sh_max);
  if (threadIdx.x == 0) scr.partials[blockIdx.x] = from_key(top);
  if (!last_block(scr.counter)) return;
  top = kKeyMin;
  for (int b = threadIdx.x; b < (int)gridDim.x; b += kReduceThreads)
    top = max(top, order_key(__ldcg(scr.partials + b)));
  top = block_max(top, sh_max);
  if (threadIdx.x == 0) {
    scr.result[0] = from_key(top);
    scr.result[3] = (double)n;
    *scr.counter = 0u;
  }
}

// a CTA's sums by a binary tree over its threads, the CTAs' sums one after another: the sum of
// the weights by one thread, of their squares by a thread on another SM quarter
__global__ void __launch_bounds__(kReduceThreads) ordered_sum_kernel(int64_t n, const double* ll, const double* lp,
                                                                     const double* lq, double* w, ReduceScratch scr) {
  __shared__ double sh[2][kReduceThreads];
  const int t = threadIdx.x;
  const int64_t stride = (int64_t)gridDim.x * kReduceThreads;
  const double m = scr.result[0];
  const bool any = order_key(m) > kKeyMin;
  double s1 = 0.0, s2 = 0.0;
  for (int64_t i = (int64_t)blockIdx.x * kReduceThreads + t; i < n; i += stride) {
    const double e = any ? exp(log_weight(ll, lp, lq, i) - m) : 0.0;
    s1 += e;
    s2 = fma(e, e, s2);
    w[i] = e;
  }
  sh[0][t] = s1;
  sh[1][t] = s2;
#pragma unroll
  for (int h = kReduceThreads / 2; h >= 32; h >>= 1) {
    __syncthreads();
    if (t < h) {
      sh[0][t] = s1 = s1 + sh[0][t + h];
      sh[1][t] = s2 = s2 + sh[1][t + h];
    }
  }
  if (t < 32) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      s1 += __shfl_xor_sync(0xffffffffu, s1, o);
      s2 += __shfl_xor_sync(0xffffffffu, s2, o);
    }
  }
  if (t == 0) {
    scr.partials[2 * blockIdx.x] = s1;
    scr.partials[2 * blockIdx.x + 1] = s2;
  }
  if (!last_block(scr.counter)) return;
  if (t == 0 || t == 32) {
    const double* p = scr.partials + (t >> 5);
    double s = 0.0;
    constexpr int kAhead = 16;
    for (int b0 = 0; b0 < (int)gridDim.x; b0 += kAhead) {
      double v[kAhead];
#pragma unroll
      for (int k = 0; k < kAhead; ++k) v[k] = b0 + k < (int)gridDim.x ? __ldcg(p + 2 * (b0 + k)) : 0.0;
#pragma unroll
      for (int k = 0; k < kAhead; ++k) s += v[k];
    }
    scr.result[1 + (t >> 5)] = s;
    if (t == 0) *scr.counter = 0u;
  }
}

__global__ void __launch_bounds__(kReduceThreads) ordered_weights_kernel(int64_t n, ReduceScratch scr, double* w) {
  const bool any = order_key(scr.result[0]) > kKeyMin;
  const double inv = 1.0 / scr.result[1];
  const int64_t stride = (int64_t)gridDim.x * kReduceThreads;
  for (int64_t i = (int64_t)blockIdx.x * kReduceThreads + threadIdx.x; i < n; i += stride)
    w[i] = any ? w[i] * inv : 0.0;
}

unsigned reduce_grid(int64_t n) {
  return (unsigned)std::max<int64_t>(1, std::min<int64_t>((n + kReduceThreads - 1) / kReduceThreads, kReduceBlocks));
}

}  // namespace

// Weights whose bits are pinned: library exponentials about the batch's maximum, every sum in a
// fixed order.  A refit feeds its moments back into the next draws, whose FP32 likelihoods turn
// a last-bit difference of a weight into one of 1e-6 in the fitted Gaussian (seen on one event
// of a dozen): with pinned sums a seed keeps its proposals.  The price is the serial sum of the
// CTAs' partials.
cudaError_t launch_reduce_ordered(int64_t n, const double* loglike, const double* logp, const double* logq,
                                  double* weights, const ReduceScratch& scr, cudaStream_t s) {
  const unsigned grid = reduce_grid(n);
  ordered_max_kernel<<<grid, kReduceThreads, 0, s>>>(n, loglike, logp, logq, scr);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  ordered_sum_kernel<<<grid, kReduceThreads, 0, s>>>(n, loglike, logp, logq, weights, scr);
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  ordered_weights_kernel<<<grid, kReduceThreads, 0, s>>>(n, scr, weights);
  return cudaGetLastError();
}

cudaError_t launch_reduce(int64_t n, const double* loglike, const double* logp, const double* logq, double* weights,
                          const ReduceScratch& scr, cudaStream_t s) {
  // one sample per thread until every CTA slot is taken: the exponentials of a small batch
  // then spread over all SMs
  const unsigned grid = reduce_grid(n);
  reduce_kernel<<<grid, kReduceThreads, 0, s>>>(n, loglike, logp, logq, weights, scr);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess || weights == nullptr) return e;
  weights_kernel<<<grid, kReduceThreads, 0, s>>>(n, scr, weights);
  return cudaGetLastError();
}

}  // namespace mbis
