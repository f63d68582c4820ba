// ga_strip_tasks.cuh -- the task list of the strip kernels (ga_strip.cuh).
#pragma once

#include "ga_strip.cuh"

namespace ga {

// Zeroed by the caller.
struct KXTaskScratch {
  unsigned long long rows;       // edge words handed out
  int32_t pairs[kKxMaxStrips];   // [k]: pairs of k + 1 strips
};
static_assert(sizeof(KXTaskScratch) % 8 == 0, "followed by edge words");

struct KXTaskParams {
  const int64_t *q_off, *t_off;
  const int32_t *sorted, *range;
  int64_t nt, q0;
  int32_t W;            // columns of a strip
  KXTaskScratch *scratch;
  KXPairState *state;   // per list entry; nstrips is set
  int2 *tasks;
  int64_t *edge_off;    // per list entry
  int32_t *ntasks;      // their number (nullable)
};

// v of thread t becomes the sum of the values of threads t.. (1,024 threads).
__device__ __forceinline__ int kx_suffix_sum(int v, int *warp_sums) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  auto in_warp = [&](int s) {
#pragma unroll
    for (int off = 1; off < 32; off *= 2) {
      const int x = __shfl_down_sync(0xffffffffu, s, off);
      if (lane + off < 32) s += x;
    }
    return s;
  };
  v = in_warp(v);
  __syncthreads();
  if (lane == 0) warp_sums[warp] = v;
  __syncthreads();
  const int w = in_warp(warp_sums[lane]);
  const int after = __shfl_sync(0xffffffffu, w, (warp + 1) & 31);
  return v + (warp < 31 ? after : 0);
}

// The pairs' strips and their counts, and the edge buffers of the pairs of more than
// one strip one after another.
__global__ void __launch_bounds__(256) kx_count_kernel(const __grid_constant__ KXTaskParams p) {
  const int i = blockIdx.x * 256 + threadIdx.x, lane = threadIdx.x & 31;
  int R = 0, ns = 0;
  if (i < p.range[1] - p.range[0]) {
    const int pid = p.sorted[p.range[0] + i];
    const int64_t qi = p.nt ? p.q0 + pid / p.nt : pid, ti = p.nt ? pid % p.nt : pid;
    const int m = (int)(p.q_off[qi + 1] - p.q_off[qi]), nn = (int)(p.t_off[ti + 1] - p.t_off[ti]);
    R = ::min(m, nn);
    ns = ::min((::max(m, nn) + p.W - 1) / p.W, kKxMaxStrips);
    p.state[i].nstrips = ns;
  }
  const unsigned peers = __match_any_sync(0xffffffffu, ns);
  if (ns > 0 && lane == __ffs(peers) - 1) atomicAdd(&p.scratch->pairs[ns - 1], __popc(peers));
  const unsigned long long own = ns > 1 ? (unsigned long long)R + 1 : 0;
  unsigned long long sum = own, first = 0;
#pragma unroll
  for (int off = 1; off < 32; off *= 2) {
    const unsigned long long x = __shfl_up_sync(0xffffffffu, sum, off);
    if (lane >= off) sum += x;
  }
  if (lane == 31 && sum) first = atomicAdd(&p.scratch->rows, sum);
  first = __shfl_sync(0xffffffffu, first, 31);
  if (ns > 0) p.edge_off[i] = ns > 1 ? (int64_t)(first + sum - own) : 0;
}

// Every strip of every listed pair, the strips with the most strips still to come
// after them first (so the longest chain of strips starts first, and a strip always
// comes after its left neighbour), otherwise roughly in list order (longest first).
// One block, for that order's sake (places taken by many blocks at once left long
// pairs to the end: 12,000 protein pairs 783 -> 868 us): what it reads of a pair is
// one word, loaded a turn ahead.  With the pairs' offsets read here twice and a scan
// by one thread it took 57 us for 6,000 pairs, now 11 with the counts: 6,000 protein
// pairs 735 -> 694 us, 12,000 1,050 -> 946, 16 queries x 8,000 targets in global mode
// 10.9 -> 7.6 ms.
__global__ void __launch_bounds__(1024) kx_tasks_kernel(const __grid_constant__ KXTaskParams p) {
  static_assert(kKxMaxStrips == 1024, "a class per thread");
  __shared__ int32_t place[kKxMaxStrips];
  __shared__ int warp_sums[32];
  const int tid = threadIdx.x, lane = tid & 31;
  const int n = p.range[1] - p.range[0];
  int next = tid < n ? p.state[tid].nstrips : 0;
  // pairs of at least k strips; a class begins after the tasks with more to go
  const int at_least = kx_suffix_sum(p.scratch->pairs[tid], warp_sums);
  const int end = kx_suffix_sum(at_least, warp_sums);
  place[tid] = end - at_least;
  if (tid == 0 && p.ntasks) *p.ntasks = end;
  __syncthreads();
  for (int i0 = 0; i0 < n; i0 += 1024) {
    const int ns = next;
    next = i0 + 1024 + tid < n ? p.state[i0 + 1024 + tid].nstrips : 0;
    for (int k = (int)__reduce_max_sync(0xffffffffu, (unsigned)ns); k >= 1; --k) {
      const unsigned in = __ballot_sync(0xffffffffu, ns >= k);
      int at = 0;
      if (lane == 0) at = atomicAdd(&place[k - 1], __popc(in));
      at = __shfl_sync(0xffffffffu, at, 0) + __popc(in & ((1u << lane) - 1));
      if (ns >= k) p.tasks[at] = make_int2(i0 + tid, ns - k);
    }
  }
}

// Both, for up to n listed pairs.
inline cudaError_t launch_kx_tasks(const KXTaskParams &p, int64_t n, cudaStream_t s) {
  kx_count_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(p);
  kx_tasks_kernel<<<1, 1024, 0, s>>>(p);
  return cudaGetLastError();
}

}  // namespace ga
