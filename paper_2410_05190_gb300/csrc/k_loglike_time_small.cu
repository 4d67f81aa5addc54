// k_loglike_time_small.cu -- the time-marginalised likelihood on tiles of 64 and 32 samples (a
// unit of its own: the instantiations compile beside those of k_loglike_time.cu).
#include "loglike_time.cuh"

namespace mbis {

cudaError_t launch_loglike_mixed_time_small(const LikeArgs& a, int32_t tile, cudaStream_t s) {
  return tile == 32 ? launch_rows<true, 32>(a, s) : launch_rows<true, 64>(a, s);
}

}  // namespace mbis
