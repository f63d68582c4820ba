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

constexpr int kKxLag = 115;                // rows a strip runs behind its left neighbour
constexpr int kKxMaxStrips = 1024;         // strips of one pair (the task order's buckets)
constexpr int64_t kKxMaxTasks = 1 << 30;   // strips of one launch (int32 places in its task list)

// Rows from the first of a pair's first strip to the last of its last, at width w.
__host__ __device__ inline int64_t kx_chain(int64_t shorter, int64_t longer, int w) {
  return shorter + kKxLag * (longer / kx_width(w));
}

// Sizes of a strip launch over a set of pairs: sum of (shorter sequence + 1), and for
// every width the strips and the edge words (the same sum over the pairs of more than
// one strip) in 64 bits each, because a search of one query of 200,000 residues against
// 11 million targets has 8.6e9 strips of 256 columns; and the longest chain.
struct LongSums {
  unsigned long long rows;
  unsigned long long strips[kKxWidths];
  unsigned long long words[kKxWidths];
  int32_t chain[kKxWidths], pad;
};

// Whether a strip launch of a tile takes these sizes: the strips of the longest
// sequence, all strips, and edge words of max_words at most.
inline bool kx_fits(int tile, int64_t longest, int64_t ntasks, int64_t words, int64_t max_words) {
  return longest <= 64 * (int64_t)kKxTileK[tile] * kKxMaxStrips && ntasks <= kKxMaxTasks && words <= max_words;
}

// The tile of a launch with strips[w] strips at width w and a longest chain of
// chain[w] rows: the one with the least estimated time.
//
// The strips of a pair move at the pace of the slowest of them, so a launch takes the
// longest chain (kx_chain: rows and lag) x the row step of a scheduler that holds
// ceil(strips / schedulers) warps.  A lone warp's step is a latency, several
// warps' the issue of their columns; both grow with K, the lag falls with it.
// Measured on GB300 (cycles per row at one warp, and more per further one).
// *cycles (nullable): the estimate.
int kx_choose(int mode, bool profile, const int64_t *chain, const int64_t *strips, int nsm, double *cycles = nullptr);

// One launch of a mode's strip kernel, or (occ != null) its blocks per SM.
cudaError_t launch_kx_local(int tile, const KXParams &p, int grid, cudaStream_t s, int *occ);
cudaError_t launch_kx_global(int tile, const KXParams &p, int grid, cudaStream_t s, int *occ);
cudaError_t launch_kx_semi(int tile, const KXParams &p, int grid, cudaStream_t s, int *occ);
inline cudaError_t launch_kx(int mode, int tile, const KXParams &p, int grid, cudaStream_t s, int *occ = nullptr) {
  return mode == 0 ? launch_kx_local(tile, p, grid, s, occ) : mode == 1 ? launch_kx_global(tile, p, grid, s, occ)
                                                                        : launch_kx_semi(tile, p, grid, s, occ);
}

}  // namespace ga
