// ga_kx_launch.cuh -- launch and occupancy of the strip kernels of one mode.
#pragma once

#include "ga_kx.h"
#include "ga_strip.cuh"

namespace ga {

// (A kernel's shared-memory limit is one setting per device for every host thread: it
// is set to the largest alphabet's profile, so that no call lowers it below what
// another one is about to launch with.)
template <int MODE, int K, bool FC, bool PROF>
cudaError_t kx_launch(const KXParams &p, int grid, cudaStream_t s, int *occ) {
  constexpr size_t largest = (size_t)kKxWarps * 32 * kx_prof_row<K>;
  const size_t smem = PROF ? (size_t)kKxWarps * (size_t)(p.A + 1) * kx_prof_row<K> : 0;
  if (PROF && largest > 40 * 1024) {
    const cudaError_t e = cudaFuncSetAttribute(kx_kernel<MODE, K, FC, PROF>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               (int)largest);
    if (e != cudaSuccess) return e;
  }
  if (occ) return cudaOccupancyMaxActiveBlocksPerMultiprocessor(occ, kx_kernel<MODE, K, FC, PROF>, 32 * kKxWarps, smem);
  kx_kernel<MODE, K, FC, PROF><<<grid, 32 * kKxWarps, smem, s>>>(p);
  return cudaGetLastError();
}

// occ != null: occupancy instead of a launch.
template <int MODE, bool PROF>
cudaError_t kx_tile(int tile, const KXParams &p, int grid, cudaStream_t s, int *occ) {
  constexpr bool kFc = MODE != kModeSemi;
  if (tile == kKx4) return kx_launch<MODE, 4, kFc, PROF>(p, grid, s, occ);
  if (tile == kKx8) return kx_launch<MODE, 8, kFc, PROF>(p, grid, s, occ);
  if constexpr (PROF) {
    if constexpr (kFc)
      if (tile == kKx8Wide) return kx_launch<MODE, 8, false, PROF>(p, grid, s, occ);
  } else {
    if (tile == kKx12) return kx_launch<MODE, 12, kFc, PROF>(p, grid, s, occ);
    if (tile == kKx16Wide) return kx_launch<MODE, 16, false, PROF>(p, grid, s, occ);
    if constexpr (kFc) {
      if (tile == kKx16) return kx_launch<MODE, 16, kFc, PROF>(p, grid, s, occ);
      if (tile == kKx20) return kx_launch<MODE, 20, kFc, PROF>(p, grid, s, occ);
    }
  }
  return cudaErrorInvalidValue;
}

}  // namespace ga

#define GA_KX_DEFINE(NAME, MODE)                                                                          \
  cudaError_t launch_kx_##NAME(int tile, const KXParams &p, int grid, cudaStream_t s, int *occ) {         \
    return p.A > 4 ? kx_tile<MODE, true>(tile, p, grid, s, occ) : kx_tile<MODE, false>(tile, p, grid, s, occ); \
  }
