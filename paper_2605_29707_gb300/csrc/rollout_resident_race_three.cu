// rollout_resident_race_three.cu -- the resident kernel's three-phase steps: the exponential race.
#include "rollout_kernels.cuh"

namespace dm {

DM_ROLL_LAUNCH(launch_resident_race_three) { return launch_resident<true, false>(p, grid, smem, stream, tm); }

}  // namespace dm
