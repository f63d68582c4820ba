// ga_strip_tasks.cuh -- the task list of the strip kernels (ga_strip.cuh).
#pragma once

#include "ga_strip.cuh"

namespace ga {

struct KXTaskParams {
  const int64_t *q_off, *t_off;
  const int32_t *sorted, *range;
  int64_t nt, q0;
  int32_t W;            // columns of a strip
  int2 *tasks;
  int64_t *edge_off;    // per list entry
  int32_t *ntasks;      // their number (nullable)
};

// One block: every strip of every listed pair, the strips with the most strips
// still to come after them first (so the longest chain of strips starts first,
// and a strip always comes after its left neighbour); edge buffers of the pairs
// of more than one strip one after another.
__global__ void kx_tasks_kernel(const __grid_constant__ KXTaskParams p) {
  __shared__ int32_t start[kKxMaxStrips + 2], cursor[kKxMaxStrips + 2];
  __shared__ unsigned long long rows;
  const int n = p.range[1] - p.range[0];
  for (int k = threadIdx.x; k < kKxMaxStrips + 2; k += blockDim.x) start[k] = cursor[k] = 0;
  if (threadIdx.x == 0) rows = 0;
  __syncthreads();
  auto strips_of = [&](int i, int &R) -> int {
    const int pid = p.sorted[p.range[0] + i];
    const int64_t qi = p.nt ? p.q0 + pid / p.nt : pid, ti = p.nt ? pid % p.nt : pid;
    const int m = (int)(p.q_off[qi + 1] - p.q_off[qi]), nn = (int)(p.t_off[ti + 1] - p.t_off[ti]);
    R = ::min(m, nn);
    return ::min((::max(m, nn) + p.W - 1) / p.W, kKxMaxStrips);
  };
  // start[k]: pairs of exactly k strips
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    int R;
    const int ns = strips_of(i, R);
    const unsigned peers = __match_any_sync(__activemask(), ns);
    if ((threadIdx.x & 31) == __ffs(peers) - 1) atomicAdd(&start[ns], __popc(peers));
    p.edge_off[i] = ns > 1 ? (int64_t)atomicAdd(&rows, (unsigned long long)(R + 1)) : 0;
  }
  __syncthreads();
  // first task with k strips to go: the tasks with more of them come before,
  // one per pair of at least that many strips
  if (threadIdx.x == 0) {
    int at_least = 0, at = 0;
    for (int k = kKxMaxStrips; k >= 1; --k) {
      at_least += start[k];
      start[k] = at;
      at += at_least;
    }
    if (p.ntasks) *p.ntasks = at;
  }
  __syncthreads();
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    int R;
    const int ns = strips_of(i, R);
    for (int k = ns; k >= 1; --k) {
      const unsigned peers = __match_any_sync(__activemask(), k);
      const int leader = __ffs(peers) - 1, lane = threadIdx.x & 31;
      int at = 0;
      if (lane == leader) at = atomicAdd(&cursor[k], __popc(peers));
      at = __shfl_sync(peers, at, leader) + __popc(peers & ((1u << lane) - 1));
      p.tasks[start[k] + at] = make_int2(i, ns - k);
    }
  }
}

}  // namespace ga
