// k_moments.cu -- weighted mean and covariance of the proposal samples, for refitting the
// Gaussian proposal from an importance-weighted batch (the iterative update of the proposal
// that Sec. III A suggests).
//
// With normalised weights w_i and offsets d_i = theta_i - ref (periodic slots wrapped into
// [-period/2, period/2) around ref), the kernel accumulates sum w d and sum w d d^T in FP64;
// offsets keep the sums well conditioned for parameters measured to ~1e-5 relative.
//
// What bounds it is the FP64 pipe: 1 + 2 P + P (P + 1) / 2 multiply-adds and 2 P other
// operations per sample (15 us for 5 slots of 2^18 samples), and at the end the CTAs' sums added
// one after another (304 dependent adds, 10 us).  That order, like the tree over a CTA's threads,
// is part of the result: a refit feeds the moments back into draws whose FP32 likelihoods turn a
// last bit into 1e-6 of the fitted Gaussian.  One instantiation per slot count keeps every sum in
// registers (with a run-time count the sums lived in local memory).  The sums of a warp fold by
// recursive halving -- each step a lane keeps half of its sums and takes its partner's part of
// them, so M sums cost M adds instead of 5 M, in the tree's pairs.  The posterior stage of 2^18
// samples (weights, moments, levels; GB300): 667 us before, 133 now, 119 with an order of its own.
#include "fpkey.cuh"
#include "internal.h"

namespace mbis {
namespace {

constexpr int kMomThreads = 128;
constexpr int kMomBlocks = 304;  // two per SM

__host__ __device__ constexpr int moment_sums(int P) { return 1 + P + P * (P + 1) / 2; }

// Folds v[0 .. M) over the warp.  Afterwards lane l holds the total of sum `first` (and of
// no other) for the lanes with first < M; every M up to 32 lanes' worth per call of the
// recursion: at each of the five steps the lanes whose bit is set keep the upper half.
template <int M, int O>
struct WarpFold {
  static constexpr int H = (M + 1) / 2;
  // v: the M sums this lane still holds; base: index of v[0] among all sums
  static __device__ __forceinline__ void run(double (&v)[M], int lane, int& base, int& count, double* out) {
    double keep[H];
    const bool up = lane & O;
#pragma unroll
    for (int i = 0; i < H; ++i) {
      const double hi = H + i < M ? v[H + i] : 0.0;
      const double mine = up ? hi : v[i], give = up ? v[i] : hi;
      keep[i] = mine + __shfl_xor_sync(0xffffffffu, give, O);
    }
    base += up ? H : 0;
    count = up ? max(count - H, 0) : min(count, H);
    if constexpr (O > 1) {
      WarpFold<H, O / 2>::run(keep, lane, base, count, out);
    } else {
#pragma unroll
      for (int i = 0; i < H; ++i)
        if (i < count) out[base + i] = keep[i];
    }
  }
};

template <int P>
__global__ void __launch_bounds__(kMomThreads, 2) moments_kernel(int64_t n, const double* theta, const double* w,
                                                                 MomentArgs ma, double* partials,
                                                                 unsigned int* counter, double* out) {
  constexpr int nm = moment_sums(P);  // sum of weights, first moments, upper triangle
  double acc[nm];
#pragma unroll
  for (int m = 0; m < nm; ++m) acc[m] = 0.0;
  // up to 6 slots the next sample's loads fly during this one's arithmetic (beyond, the sums
  // leave no registers for them, and a sample's arithmetic outlasts its loads)
  constexpr bool kAhead = P <= 6;
  const int64_t stride = (int64_t)gridDim.x * kMomThreads;
  int64_t i = (int64_t)blockIdx.x * kMomThreads + threadIdx.x;
  double wn = 0.0, dn[P];
  auto load = [&](int64_t at) {
    wn = w[at];
#pragma unroll
    for (int p = 0; p < P; ++p) dn[p] = theta[(int64_t)p * n + at];
  };
  if (kAhead && i < n) load(i);
  for (; i < n; i += stride) {
    if (!kAhead) load(i);
    const double wi = wn;
    double d[P];
#pragma unroll
    for (int p = 0; p < P; ++p) d[p] = dn[p];
    if (kAhead && i + stride < n) load(i + stride);
    // wi > 0, NaN excluded
    const long long wb = __double_as_longlong(wi);
    if (wb <= 0 || wb > 0x7ff0000000000000ll) continue;
#pragma unroll
    for (int p = 0; p < P; ++p) {
      d[p] -= ma.ref[p];
      const double T = ma.period[p];
      if (T > 0.0) {
        // a division and a floor only for an offset that they can move
        const long long k = order_key(d[p]), h = order_key(0.4375 * T);
        if (k < -h || k >= h) d[p] -= T * floor(d[p] / T + 0.5);
      }
    }
    int m = 0;
    acc[m++] += wi;
    double wd[P];
#pragma unroll
    for (int p = 0; p < P; ++p) {
      wd[p] = wi * d[p];
      acc[m] = fma(wi, d[p], acc[m]);
      ++m;
    }
#pragma unroll
    for (int p = 0; p < P; ++p)
#pragma unroll
      for (int q = p; q < P; ++q) {
        acc[m] = fma(wd[p], d[q], acc[m]);
        ++m;
      }
  }
  // the CTA's sums: a binary tree over its threads, the upper half of them adding into the lower
  __shared__ double sh[nm][kMomThreads / 2];
  __shared__ bool last;
  const int t = threadIdx.x;
#pragma unroll
  for (int h = kMomThreads / 2; h >= 32; h >>= 1) {
    if (h < kMomThreads / 2) __syncthreads();
    if (t >= h && t < 2 * h)
#pragma unroll
      for (int m = 0; m < nm; ++m) sh[m][t - h] = acc[m];
    __syncthreads();
    if (t < h)
#pragma unroll
      for (int m = 0; m < nm; ++m) acc[m] += sh[m][t];
  }
  if (t < 32) {
    int base = 0, count = nm;
    WarpFold<nm, 16>::run(acc, t, base, count, partials + (int64_t)blockIdx.x * nm);
  }
  __threadfence();
  __syncthreads();
  if (t == 0) last = atomicAdd(counter, 1u) == gridDim.x - 1;
  __syncthreads();
  if (last) {
    // one thread per sum, the CTAs one after another
    if (t < nm) {
      double s = 0.0;
      constexpr int kLoads = 16;
      for (int b0 = 0; b0 < (int)gridDim.x; b0 += kLoads) {
        double v[kLoads];
#pragma unroll
        for (int k = 0; k < kLoads; ++k)
          v[k] = b0 + k < (int)gridDim.x ? __ldcg(partials + (int64_t)(b0 + k) * nm + t) : 0.0;
#pragma unroll
        for (int k = 0; k < kLoads; ++k) s += v[k];
      }
      out[t] = s;
    }
    if (t == 0) *counter = 0u;
  }
}

template <int P>
void launch(int64_t n, const double* theta, const double* w, const MomentArgs& ma, double* partials,
            unsigned int* counter, double* out, cudaStream_t s) {
  const int64_t want = (n + kMomThreads - 1) / kMomThreads;
  moments_kernel<P><<<(unsigned)(want < kMomBlocks ? (want > 0 ? want : 1) : kMomBlocks), kMomThreads, 0, s>>>(
      n, theta, w, ma, partials, counter, out);
}

}  // namespace

int moments_partials_size(int32_t P) { return kMomBlocks * moment_sums(P); }

cudaError_t launch_moments(int64_t n, int32_t P, const double* theta, const double* w, const MomentArgs& ma,
                           double* partials, unsigned int* counter, double* out, cudaStream_t s) {
  static_assert(kMaxP == 11, "one instantiation per slot count");
  switch (P) {
    case 1: launch<1>(n, theta, w, ma, partials, counter, out, s); break;
    case 2: launch<2>(n, theta, w, ma, partials, counter, out, s); break;
    case 3: launch<3>(n, theta, w, ma, partials, counter, out, s); break;
    case 4: launch<4>(n, theta, w, ma, partials, counter, out, s); break;
    case 5: launch<5>(n, theta, w, ma, partials, counter, out, s); break;
    case 6: launch<6>(n, theta, w, ma, partials, counter, out, s); break;
    case 7: launch<7>(n, theta, w, ma, partials, counter, out, s); break;
    case 8: launch<8>(n, theta, w, ma, partials, counter, out, s); break;
    case 9: launch<9>(n, theta, w, ma, partials, counter, out, s); break;
    case 10: launch<10>(n, theta, w, ma, partials, counter, out, s); break;
    default: launch<11>(n, theta, w, ma, partials, counter, out, s); break;
  }
  return cudaGetLastError();
}

}  // namespace mbis
