// Scheme dispatch of the two-step launches of one storage type.
#pragma once

#include "lbm_launch.cuh"
#include "lbm_two_step.cuh"

namespace lbm {

template <class S, int SCHEME, int LAYOUT>
cudaError_t two_step_launch_one(const StripLaunch& L, int grid, cudaStream_t s) {
  two_step_kernel<S, SCHEME, LAYOUT><<<grid, kTwoThreads, 0, s>>>(make_args<S>(L));
  return cudaGetLastError();
}

template <class S, int LAYOUT>
cudaError_t two_step_launch_t(int scheme, const StripLaunch& L, int grid, cudaStream_t s) {
  switch (scheme) {
    case kSC: return two_step_launch_one<S, kSC, LAYOUT>(L, grid, s);
    case kEDM: return two_step_launch_one<S, kEDM, LAYOUT>(L, grid, s);
    case kImproved: return two_step_launch_one<S, kImproved, LAYOUT>(L, grid, s);
    case kNoForce: return two_step_launch_one<S, kNoForce, LAYOUT>(L, grid, s);
    case kEDMMod: return two_step_launch_one<S, kEDMMod, LAYOUT>(L, grid, s);
    case kLadd: return two_step_launch_one<S, kLadd, LAYOUT>(L, grid, s);
    case kMRT: return two_step_launch_one<S, kMRT, LAYOUT>(L, grid, s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace lbm
