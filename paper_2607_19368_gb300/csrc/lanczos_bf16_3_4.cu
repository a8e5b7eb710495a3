// Lanczos kernel instantiations for 3 float4 column groups of Phi per lane and
// 4 warps per row (D <= 1536), bfloat16 Phi, for every basis tile count KT.
#include "lanczos_kernel.cuh"

namespace sls {

int launch_lanczos_bf16_3_4(SLS_LZ_LAUNCH_ARGS) {
  return launch_lanczos_kt<3, 4, uint16_t>(SLS_LZ_PASS_ARGS);
}

}  // namespace sls
