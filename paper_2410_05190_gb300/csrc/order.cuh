// order.cuh -- a counting order of samples by a small integer key, largest key first (equal
// keys in any order): the work order of the likelihood kernels (live bins) and of the tile
// assignment (live-bin counts).
//
// Two passes over the samples around a one-CTA scan.  Each CTA counts its samples' keys in
// shared memory and adds the counts to the global ones (first pass) or reserves that many
// slots per key (second pass), so that global atomics happen once per CTA and key and not
// once per warp and key: the per-warp version took 14 and 15 us at 2^18 samples of 503 keys
// against 6.7 and 6.9 here.  Keys beyond kOrderSmemKeys keep the per-warp version.
#pragma once
#include <algorithm>

#include <cuda_runtime.h>

#include <cstdint>

namespace mbis {

constexpr int kOrderThreads = 512;
constexpr int kOrderCtas = 2 * 152;
constexpr int kOrderKeep = 8;            // samples a thread holds between counting and placing
constexpr int32_t kOrderSmemKeys = 12288;  // keys counted in shared memory (48 KB)

// Per-warp version: lanes with the same key add once per warp.
template <bool kPlace, typename Key>
__device__ __forceinline__ void order_by_warp(int64_t n, Key key, int32_t* counts, int32_t* perm) {
  const int lane = threadIdx.x & 31;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t base = (int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31); base < n; base += stride) {
    const int64_t i = base + lane;
    const bool on = i < n;
    const unsigned mask = __ballot_sync(0xffffffffu, on);
    if (on) {
      const int32_t k = key(i);
      const unsigned peers = __match_any_sync(mask, k);
      const int leader = __ffs(peers) - 1;
      int32_t first = 0;
      if (lane == leader) first = atomicAdd(&counts[k], __popc(peers));
      if constexpr (kPlace) {
        first = __shfl_sync(peers, first, leader);
        perm[first + __popc(peers & ((1u << lane) - 1u))] = (int32_t)i;
      }
    }
  }
}

// kPlace: counts holds the first free slot of each key, which the CTA's samples take;
// otherwise the CTA's counts are added to it.
template <bool kPlace, typename Key>
__global__ void __launch_bounds__(kOrderThreads) order_kernel(int64_t n, int32_t n_keys, Key key, int32_t* counts,
                                                              int32_t* perm) {
  extern __shared__ int32_t h[];
  if (n_keys > kOrderSmemKeys) {
    order_by_warp<kPlace>(n, key, counts, perm);
    return;
  }
  const int64_t stride = (int64_t)gridDim.x * kOrderThreads;
  for (int64_t base = (int64_t)blockIdx.x * kOrderThreads; base < n; base += kOrderKeep * stride) {
    for (int32_t k = threadIdx.x; k < n_keys; k += kOrderThreads) h[k] = 0;
    __syncthreads();
    int32_t my_key[kOrderKeep], my_rank[kOrderKeep];
#pragma unroll
    for (int r = 0; r < kOrderKeep; ++r) {
      const int64_t i = base + r * stride + threadIdx.x;
      my_key[r] = i < n ? key(i) : -1;
      if (my_key[r] >= 0) my_rank[r] = atomicAdd(&h[my_key[r]], 1);
    }
    __syncthreads();
    for (int32_t k = threadIdx.x; k < n_keys; k += kOrderThreads)
      if (h[k] > 0) h[k] = atomicAdd(&counts[k], h[k]);
    if constexpr (kPlace) {
      __syncthreads();
#pragma unroll
      for (int r = 0; r < kOrderKeep; ++r)
        if (my_key[r] >= 0) perm[h[my_key[r]] + my_rank[r]] = (int32_t)(base + r * stride + threadIdx.x);
    }
    __syncthreads();
  }
}

// one CTA: counts -> first slot of each key, keys in decreasing order (k_order.cu)
cudaError_t launch_order_scan(int32_t n_keys, int32_t* counts, cudaStream_t s);

// perm[slot] = sample, largest key first; counts (n_keys ints) and perm (n ints) are the
// caller's scratch, key(i) in [0, n_keys)
template <typename Key>
cudaError_t launch_order(int64_t n, int32_t n_keys, const Key& key, int32_t* counts, int32_t* perm, cudaStream_t s) {
  cudaError_t e = cudaMemsetAsync(counts, 0, sizeof(int32_t) * (size_t)n_keys, s);
  if (e != cudaSuccess) return e;
  const unsigned grid =
      (unsigned)std::max<int64_t>(1, std::min<int64_t>((n + kOrderThreads - 1) / kOrderThreads, kOrderCtas));
  const size_t smem = n_keys > kOrderSmemKeys ? 0 : sizeof(int32_t) * (size_t)n_keys;
  order_kernel<false><<<grid, kOrderThreads, smem, s>>>(n, n_keys, key, counts, perm);
  e = launch_order_scan(n_keys, counts, s);
  if (e != cudaSuccess) return e;
  order_kernel<true><<<grid, kOrderThreads, smem, s>>>(n, n_keys, key, counts, perm);
  return cudaGetLastError();
}

}  // namespace mbis
