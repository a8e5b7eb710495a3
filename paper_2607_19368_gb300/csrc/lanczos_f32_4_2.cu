// Lanczos kernel instantiations for 4 float4 column groups of Phi per lane and
// 2 warps per row (D <= 1024), float32 Phi, for every basis tile count KT.
#include "lanczos_kernel.cuh"

namespace sls {

int launch_lanczos_f32_4_2(SLS_LZ_LAUNCH_ARGS) {
  return launch_lanczos_kt<4, 2, float>(SLS_LZ_PASS_ARGS);
}

}  // namespace sls
