// rollout_resident_fast.cu -- the resident kernel's one-barrier steps: greedy and inverse-CDF loops.
#include "rollout_kernels.cuh"

namespace dm {

DM_ROLL_LAUNCH(launch_resident_fast) { return launch_resident<false, true>(p, grid, smem, stream, tm); }

DM_ROLL_LAUNCH(launch_rollout_cdf_mma) {
  if (p.B == 1)
    return launch_coop(rollout_resident_kernel<1, true, false, true, true>, p, grid, kRollThreads, smem, stream, tm);
  if (p.B == 2)
    return launch_coop(rollout_resident_kernel<2, true, false, true, true>, p, grid, kRollThreads, smem, stream, tm);
  return cudaErrorInvalidValue;
}

}  // namespace dm
