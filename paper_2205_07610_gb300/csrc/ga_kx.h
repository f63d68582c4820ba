// ga_kx.h -- host side of the strip kernels (ga_strip.cuh).
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

namespace ga {

struct KXParams;

// Strip widths: 64 K columns for K = 4, 8, 12, 16, 20.
constexpr int kKxWidths = 5;
constexpr __host__ __device__ int kx_width(int w) { return 256 * (w + 1); }

// Column tiles: columns per lane and half, with the one-op column chain (except
// in semi-global mode) or, the last two, without it.
enum KxTile { kKx4 = 0, kKx8, kKx12, kKx16, kKx20, kKx8Wide, kKx16Wide, kKxTiles };
constexpr int kKxTileK[kKxTiles] = {4, 8, 12, 16, 20, 8, 16};

// The tile of a launch with strips[w] strips at width w whose longest pair has
// `longest` rows: the one with the least estimated time.
//
// The strips of a pair move at the pace of the slowest of them, so a launch takes
// (rows + 115 rows of lag per strip) x the row step of a scheduler that holds
// ceil(strips / schedulers) warps.  A lone warp's step is a latency, several
// warps' the issue of their columns; both grow with K, the lag falls with it.
// Measured on GB300 (cycles per row at one warp, and more per further one).
// *cycles (nullable): the estimate.
int kx_choose(int mode, bool profile, int64_t longest, const int64_t *strips, int nsm, double *cycles = nullptr);

// One launch of a mode's strip kernel, or (occ != null) its blocks per SM.
cudaError_t launch_kx_local(int tile, const KXParams &p, int grid, cudaStream_t s, int *occ);
cudaError_t launch_kx_global(int tile, const KXParams &p, int grid, cudaStream_t s, int *occ);
cudaError_t launch_kx_semi(int tile, const KXParams &p, int grid, cudaStream_t s, int *occ);
inline cudaError_t launch_kx(int mode, int tile, const KXParams &p, int grid, cudaStream_t s, int *occ = nullptr) {
  return mode == 0 ? launch_kx_local(tile, p, grid, s, occ) : mode == 1 ? launch_kx_global(tile, p, grid, s, occ)
                                                                        : launch_kx_semi(tile, p, grid, s, occ);
}

}  // namespace ga
