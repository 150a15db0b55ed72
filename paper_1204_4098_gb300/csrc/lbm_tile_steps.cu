// Two to four time steps per launch on tiles, FP32 storage (lbm_tile_steps.cuh).
#include "lbm_tile_steps.cuh"

#include "lbm_launch.cuh"

namespace lbm {

namespace {

template <int SCHEME>
cudaError_t launch(const StripLaunch& L, int steps, int most, int grid, int threads,
                   cudaStream_t s) {
  const int smem = (kQ * kTilePlane + 2 * threads) * int(sizeof(float));
  if (smem > 48 * 1024) {
    const cudaError_t e = cudaFuncSetAttribute(
        tile_steps_kernel<SCHEME>, cudaFuncAttributeMaxDynamicSharedMemorySize,
        kTilePlanes * 2 * 32 * kTileMaxWarps * int(sizeof(float)));
    if (e != cudaSuccess) return e;
  }
  tile_steps_kernel<SCHEME><<<grid, threads, smem, s>>>(make_args<StoreF32>(L), steps,
                                                    2 * most);
  return cudaGetLastError();
}

}  // namespace

cudaError_t tile_steps_launch(int scheme, const StripLaunch& L, int steps, int most, int grid,
                              int threads, cudaStream_t s) {
  switch (scheme) {
    case kSC: return launch<kSC>(L, steps, most, grid, threads, s);
    case kEDM: return launch<kEDM>(L, steps, most, grid, threads, s);
    case kImproved: return launch<kImproved>(L, steps, most, grid, threads, s);
    case kNoForce: return launch<kNoForce>(L, steps, most, grid, threads, s);
    case kEDMMod: return launch<kEDMMod>(L, steps, most, grid, threads, s);
    case kLadd: return launch<kLadd>(L, steps, most, grid, threads, s);
    case kMRT: return launch<kMRT>(L, steps, most, grid, threads, s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace lbm
