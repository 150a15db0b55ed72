// Two time steps per launch, FP32 storage (lbm_two_step.cuh).
#include "lbm_two_step_launch.cuh"

namespace lbm {

cudaError_t two_step_launch_f32(int scheme, const StripLaunch& L, int grid, bool few,
                                cudaStream_t s) {
  return L.nx % 2 ? two_step_launch_t<StoreF32, kFlatOdd>(scheme, L, grid, few, s)
                  : two_step_launch_t<StoreF32, kFlatEven>(scheme, L, grid, few, s);
}

}  // namespace lbm
