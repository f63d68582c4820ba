// Strip kernels (ga_strip.cuh), global mode.
#include "ga_kx_launch.cuh"

namespace ga {
GA_KX_DEFINE(global, kModeGlobal)
}  // namespace ga
