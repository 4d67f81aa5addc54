// k_levels.cu -- credible level of a reference point under importance weights, the quantity
// of the P-P self-consistency test (Sec. III A): for each sampled slot, the weighted fraction
// of the samples below the reference, ties counting half.
//
// One thread-block cluster of 16 CTAs per slot: the call has no scratch and may not allocate,
// and a cluster folds its CTAs' sums through distributed shared memory.  The pass reads 16
// bytes per sample and slot; one CTA per slot, as before, kept a handful of loads in flight
// on P of the 152 SMs (461 us for 5 slots of 2^18 samples, device time).  16 CTAs of 512
// threads with the next four samples of a thread in flight during the adds of these, one FP64
// add per sample, and the two sums of a warp folded by its two halves take 24 us (27 without
// the loads ahead and with a fold each).  Sums are FP64 in a fixed order (deterministic).  Sixteen
// is beyond the portable cluster size: where it cannot be placed (a partition of the GPU) the
// launch is refused, and one of eight, then of a single CTA per slot, takes its place.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <cmath>

#include "fpkey.cuh"
#include "internal.h"

namespace mbis {
namespace {

constexpr int kLevelThreads = 512;
constexpr int kLevelUnroll = 4;
constexpr int kMaxLevelSlots = 16;
static_assert(kLevelThreads == 16 * 32, "half a warp folds the CTA's warps");

struct LevelRef {
  double r[kMaxLevelSlots];
};

// kCtas: CTAs per slot, a cluster of at most 16 (half a warp folds them)
template <int kCtas>
__global__ void __launch_bounds__(kLevelThreads) levels_kernel(int64_t n, const double* __restrict__ theta,
                                                               const double* __restrict__ w,
                                                               const __grid_constant__ LevelRef ref,
                                                               double* __restrict__ out) {
  namespace cg = cooperative_groups;
  cg::cluster_group cluster = cg::this_cluster();
  __shared__ double s_warp[2][kLevelThreads / 32], s_cta[2];
  const int p = blockIdx.x / kCtas, rank = blockIdx.x % kCtas, lane = threadIdx.x & 31;
  const long long r = order_key(ref.r[p]);
  const bool r_nan = is_nan(ref.r[p]);
  const double* x = theta + (int64_t)p * n;
  double below = 0.0, above = 0.0;
  constexpr int64_t kStride = (int64_t)kCtas * kLevelThreads;
  double wn[kLevelUnroll], xn[kLevelUnroll];
  auto load = [&](int64_t i0) {
#pragma unroll
    for (int u = 0; u < kLevelUnroll; ++u) {
      const int64_t i = i0 + u * kStride;
      wn[u] = i < n ? w[i] : 0.0;
      xn[u] = i < n ? x[i] : 0.0;
    }
  };
  int64_t i0 = (int64_t)rank * kLevelThreads + threadIdx.x;
  load(i0);
  while (i0 < n) {
    double wi[kLevelUnroll], xi[kLevelUnroll];
#pragma unroll
    for (int u = 0; u < kLevelUnroll; ++u) {
      wi[u] = wn[u];
      xi[u] = xn[u];
    }
    i0 += kLevelUnroll * kStride;
    load(i0);  // the next samples' loads fly during these ones' adds
#pragma unroll
    for (int u = 0; u < kLevelUnroll; ++u) {
      // one FP64 add per sample: to the weight below or to the rest (a NaN is not below)
      if (order_key(wi[u]) <= 0 || is_nan(wi[u])) continue;
      const long long k = order_key(xi[u]);
      const bool nan = r_nan || is_nan(xi[u]);
      if (k == r && !nan) {  // a tie counts half
        below += 0.5 * wi[u];
        above += 0.5 * wi[u];
        continue;
      }
      const bool lt = k < r && !nan;
      const double sum = (lt ? below : above) + wi[u];
      below = lt ? sum : below;
      above = lt ? above : sum;
    }
  }
  // the lower half of a warp folds the weight below, the upper half the total: one add a step
  const int half = lane >> 4, hl = lane & 15;
  const double tot = below + above;
  double v = (half ? tot : below) + __shfl_xor_sync(0xffffffffu, half ? below : tot, 16);
  auto fold16 = [&] {
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  };
  fold16();
  if (hl == 0) s_warp[half][threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x < 32) {
    v = s_warp[half][hl];
    fold16();
    if (hl == 0) s_cta[half] = v;
  }
  cluster.sync();
  if (rank == 0 && threadIdx.x < 32) {
    v = hl < kCtas ? cluster.map_shared_rank(s_cta, hl)[half] : 0.0;
    fold16();
    const double all = __shfl_sync(0xffffffffu, v, 16);
    if (lane == 0) out[p] = all > 0.0 ? v / all : NAN;
  }
  cluster.sync();  // a CTA's shared memory outlives the reads of rank 0
}

template <int kCtas>
cudaError_t launch(int64_t n, int32_t P, const double* theta, const double* w, const LevelRef& ref, double* out,
                   cudaStream_t s) {
  cudaError_t e = cudaFuncSetAttribute(levels_kernel<kCtas>, cudaFuncAttributeNonPortableClusterSizeAllowed, kCtas > 8);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(P * kCtas));
  cfg.blockDim = dim3(kLevelThreads);
  cfg.stream = s;
  cudaLaunchAttribute attr = {};
  attr.id = cudaLaunchAttributeClusterDimension;
  attr.val.clusterDim.x = kCtas;
  attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  e = cudaLaunchKernelEx(&cfg, levels_kernel<kCtas>, n, theta, w, ref, out);
  const cudaError_t sticky = cudaGetLastError();
  return e != cudaSuccess ? e : sticky;
}

// with clusters of at most max_ctas CTAs
cudaError_t launch_levels(int64_t n, int32_t P, const double* theta, const double* w, const LevelRef& ref, double* out,
                          int32_t max_ctas, cudaStream_t s) {
  cudaError_t e = cudaErrorUnknown;
  if (max_ctas >= 16) e = launch<16>(n, P, theta, w, ref, out, s);
  if (e != cudaSuccess && max_ctas >= 8) e = launch<8>(n, P, theta, w, ref, out, s);
  return e == cudaSuccess ? e : launch<1>(n, P, theta, w, ref, out, s);
}

}  // namespace
}  // namespace mbis

extern "C" mbis_status mbis_debug_credible_levels(int64_t n, int32_t P, const double* theta, const double* weights,
                                                  const double* ref, double* levels, int32_t max_ctas, void* stream) {
  if (n < 1 || P < 1 || P > mbis::kMaxLevelSlots || !theta || !weights || !ref || !levels) {
    mbis::set_last_error("mbis_credible_levels: need n >= 1, 1 <= P <= 16 and non-null buffers");
    return MBIS_E_INVALID;
  }
  mbis::LevelRef r = {};
  for (int p = 0; p < P; ++p) r.r[p] = ref[p];
  const cudaError_t e =
      mbis::launch_levels(n, P, theta, weights, r, levels, max_ctas, static_cast<cudaStream_t>(stream));
  if (e != cudaSuccess) {
    mbis::set_last_error(std::string("mbis_credible_levels: ") + cudaGetErrorString(e));
    return MBIS_E_CUDA;
  }
  return MBIS_OK;
}

extern "C" mbis_status mbis_credible_levels(int64_t n, int32_t P, const double* theta, const double* weights,
                                            const double* ref, double* levels, void* stream) {
  return mbis_debug_credible_levels(n, P, theta, weights, ref, levels, 16, stream);
}
