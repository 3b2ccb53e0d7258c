// rollout_cdf.cu -- the sequential draft loop's resident kernel with phase C on the tensor cores,
// instantiated for the inverse-CDF rule (kCdf), compiled apart from rollout.cu's greedy ones.
#include "rollout_kernels.cuh"

namespace dm {

cudaError_t launch_rollout_cdf_mma(const RolloutParams& p, int grid, size_t smem, cudaStream_t stream,
                                   const CUtensorMap& tm) {
  if (p.B == 1) return launch_coop(rollout_resident_kernel<1, true, false, true>, p, grid, kRollThreads, smem, stream, tm);
  if (p.B == 2) return launch_coop(rollout_resident_kernel<2, true, false, true>, p, grid, kRollThreads, smem, stream, tm);
  return cudaErrorInvalidValue;
}

}  // namespace dm
