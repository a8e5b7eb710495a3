// Lanczos kernel instantiations for 2 float4 column groups of Phi per lane and
// 1 warp per row (D <= 256), float32 Phi, for every basis tile count KT.
#include "lanczos_kernel.cuh"

namespace sls {

int launch_lanczos_f32_2_1(SLS_LZ_LAUNCH_ARGS) {
  return launch_lanczos_kt<2, 1, float>(SLS_LZ_PASS_ARGS);
}

}  // namespace sls
