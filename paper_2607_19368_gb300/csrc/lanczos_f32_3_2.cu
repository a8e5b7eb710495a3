// Lanczos kernel instantiations for 3 float4 column groups of Phi per lane and
// 2 warps per row (D <= 768), float32 Phi, for every basis tile count KT.
#include "lanczos_kernel.cuh"

namespace sls {

int launch_lanczos_f32_3_2(SLS_LZ_LAUNCH_ARGS) {
  return launch_lanczos_kt<3, 2, float>(SLS_LZ_PASS_ARGS);
}

}  // namespace sls
