// Strip kernels (ga_strip.cuh), semi-global mode.
#include "ga_kx_launch.cuh"

namespace ga {
GA_KX_DEFINE(semi, kModeSemi)
}  // namespace ga
