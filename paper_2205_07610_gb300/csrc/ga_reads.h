// ga_reads.h -- launcher of the small-batch kernel (ga_reads.cuh).
#pragma once

#include <cuda_runtime.h>

namespace ga {

struct KRParams;
cudaError_t launch_kr(int mode, const KRParams &p, cudaStream_t s);

}  // namespace ga
