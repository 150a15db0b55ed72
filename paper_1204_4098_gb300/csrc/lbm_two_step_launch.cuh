// Scheme dispatch of the two-step launches of one storage type.
#pragma once

#include "lbm_launch.cuh"
#include "lbm_two_step.cuh"

namespace lbm {

// few: the launch brings at most kTwoFewCtas CTAs to an SM.
template <class S, int SCHEME, int LAYOUT>
cudaError_t two_step_launch_one(const StripLaunch& L, int grid, bool few, cudaStream_t s) {
  if (few)
    two_step_kernel<S, SCHEME, LAYOUT, kTwoFewCtas><<<grid, kTwoThreads, 0, s>>>(make_args<S>(L));
  else
    two_step_kernel<S, SCHEME, LAYOUT, kTwoManyCtas><<<grid, kTwoThreads, 0, s>>>(make_args<S>(L));
  return cudaGetLastError();
}

template <class S, int LAYOUT>
cudaError_t two_step_launch_t(int scheme, const StripLaunch& L, int grid, bool few,
                              cudaStream_t s) {
  switch (scheme) {
    case kSC: return two_step_launch_one<S, kSC, LAYOUT>(L, grid, few, s);
    case kEDM: return two_step_launch_one<S, kEDM, LAYOUT>(L, grid, few, s);
    case kImproved: return two_step_launch_one<S, kImproved, LAYOUT>(L, grid, few, s);
    case kNoForce: return two_step_launch_one<S, kNoForce, LAYOUT>(L, grid, few, s);
    case kEDMMod: return two_step_launch_one<S, kEDMMod, LAYOUT>(L, grid, few, s);
    case kLadd: return two_step_launch_one<S, kLadd, LAYOUT>(L, grid, few, s);
    case kMRT: return two_step_launch_one<S, kMRT, LAYOUT>(L, grid, few, s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace lbm
