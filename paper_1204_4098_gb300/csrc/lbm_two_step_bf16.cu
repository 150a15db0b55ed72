// Two time steps per launch, StoreBF16 storage (lbm_two_step.cuh).
#include "lbm_two_step_launch.cuh"

namespace lbm {

cudaError_t two_step_launch_bf16(int scheme, const StripLaunch& L, int grid, bool few,
                                 cudaStream_t s) {
  return two_step_launch_t<StoreBF16, kFlatEven>(scheme, L, grid, few, s);
}

}  // namespace lbm
