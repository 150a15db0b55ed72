// Two time steps per launch, FP32 storage (lbm_two_step.cuh).
#include "lbm_two_step.cuh"

#include "lbm_launch.cuh"

namespace lbm {

namespace {

template <int SCHEME>
cudaError_t launch(const StripLaunch& L, int grid, cudaStream_t s) {
  const StripArgs<StoreF32> A = make_args<StoreF32>(L);
  if (L.nx % 2)
    two_step_kernel<SCHEME, kFlatOdd><<<grid, kTwoThreads, 0, s>>>(A);
  else
    two_step_kernel<SCHEME, kFlatEven><<<grid, kTwoThreads, 0, s>>>(A);
  return cudaGetLastError();
}

}  // namespace

cudaError_t two_step_launch(int scheme, const StripLaunch& L, int grid, cudaStream_t s) {
  switch (scheme) {
    case kSC: return launch<kSC>(L, grid, s);
    case kEDM: return launch<kEDM>(L, grid, s);
    case kImproved: return launch<kImproved>(L, grid, s);
    case kNoForce: return launch<kNoForce>(L, grid, s);
    case kEDMMod: return launch<kEDMMod>(L, grid, s);
    case kLadd: return launch<kLadd>(L, grid, s);
    case kMRT: return launch<kMRT>(L, grid, s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace lbm
