// rollout_resident_race_fast.cu -- the resident kernel's one-barrier steps: the exponential race.
#include "rollout_kernels.cuh"

namespace dm {

DM_ROLL_LAUNCH(launch_resident_race_fast) { return launch_resident<true, true>(p, grid, smem, stream, tm); }

}  // namespace dm
