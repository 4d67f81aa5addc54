// k_loglike_time.cu -- launches of the time-marginalised likelihood (loglike_time.cuh).
#include "loglike_time.cuh"

namespace mbis {

// The samples of a tile.  A CTA's time is a chain -- set-up, then per K-block rows, MMA and
// drain -- that the number of its samples hardly shortens at two threads each, so a launch of
// fewer 128-sample tiles than SMs leaves SMs idle and the others no faster: with 64 or 32
// samples per CTA the threads of a sample share a block's bins and each warp drains fewer
// columns.  The lines lie at one CTA per SM.  Measured (us, 128 / 64 / 32 samples per CTA,
// three detectors): 3001 samples 69.6 / 55.4 / 48.2, 6000 87.0 / 74.3 / 74.8, 9000 88.5 / 75.9 /
// 80.7, 12000 89.3 / 86.4 / 114, 25000 105 / 133 / 170.  A sample's arithmetic does not depend on
// the tile.  FP64 block entry (rare: phase terms beyond 2^16 turns) keeps the large tile.
constexpr int64_t kSms = 152;

cudaError_t launch_loglike_mixed_time(const LikeArgs& a, cudaStream_t s) {
  if (a.n <= 0) return cudaSuccess;
  if (!a.ff_phase) return launch_rows<false, 128>(a, s);
  if (a.n <= 32 * kSms) return launch_loglike_mixed_time_small(a, 32, s);
  if (a.n <= 64 * kSms) return launch_loglike_mixed_time_small(a, 64, s);
  return launch_rows<true, 128>(a, s);
}

}  // namespace mbis
