// Strip kernels (ga_strip.cuh), local mode.
#include "ga_kx_launch.cuh"

namespace ga {
GA_KX_DEFINE(local, kModeLocal)
}  // namespace ga
