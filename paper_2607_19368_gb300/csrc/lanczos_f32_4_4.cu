// Lanczos kernel instantiations for 4 float4 column groups of Phi per lane and
// 4 warps per row (D <= 2048), float32 Phi, for every basis tile count KT.
#include "lanczos_kernel.cuh"

namespace sls {

int launch_lanczos_f32_4_4(SLS_LZ_LAUNCH_ARGS) {
  return launch_lanczos_kt<4, 4, float>(SLS_LZ_PASS_ARGS);
}

}  // namespace sls
