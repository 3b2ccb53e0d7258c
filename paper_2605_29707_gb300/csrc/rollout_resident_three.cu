// rollout_resident_three.cu -- the resident kernel's three-phase steps: greedy and inverse-CDF loops.
#include "rollout_kernels.cuh"

namespace dm {

DM_ROLL_LAUNCH(launch_resident_three) { return launch_resident<false, false>(p, grid, smem, stream, tm); }

}  // namespace dm
