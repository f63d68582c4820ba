// Small batches of short pairs (ga_reads.cuh).
#include "ga_reads.cuh"

#include "ga_reads.h"

namespace ga {

cudaError_t launch_kr(int mode, const KRParams &p, cudaStream_t s) {
  const int grid = (p.npairs + kKrWarps - 1) / kKrWarps;
  if (mode == kModeLocal) kr_kernel<kModeLocal><<<grid, 32 * kKrWarps, 0, s>>>(p);
  else if (mode == kModeGlobal) kr_kernel<kModeGlobal><<<grid, 32 * kKrWarps, 0, s>>>(p);
  else kr_kernel<kModeSemi><<<grid, 32 * kKrWarps, 0, s>>>(p);
  return cudaGetLastError();
}

}  // namespace ga
