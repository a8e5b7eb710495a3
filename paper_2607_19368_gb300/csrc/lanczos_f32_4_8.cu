// Lanczos kernel instantiations for 4 float4 column groups of Phi per lane and
// 8 warps per row (D <= 4096), float32 Phi, for every basis tile count KT.
#include "lanczos_kernel.cuh"

namespace sls {

int launch_lanczos_f32_4_8(SLS_LZ_LAUNCH_ARGS) {
  return launch_lanczos_kt<4, 8, float>(SLS_LZ_PASS_ARGS);
}

}  // namespace sls
