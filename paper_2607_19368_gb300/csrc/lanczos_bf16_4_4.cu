// Lanczos kernel instantiations for 4 float4 column groups of Phi per lane and
// 4 warps per row (D <= 2048), bfloat16 Phi, for every basis tile count KT.
#include "lanczos_kernel.cuh"

namespace sls {

int launch_lanczos_bf16_4_4(SLS_LZ_LAUNCH_ARGS) {
  return launch_lanczos_kt<4, 4, uint16_t>(SLS_LZ_PASS_ARGS);
}

}  // namespace sls
