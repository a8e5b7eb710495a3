// Lanczos kernel instantiations for 4 float4 column groups of Phi per lane and
// 2 warps per row (D <= 1024), bfloat16 Phi, for every basis tile count KT.
#include "lanczos_kernel.cuh"

namespace sls {

int launch_lanczos_bf16_4_2(SLS_LZ_LAUNCH_ARGS) {
  return launch_lanczos_kt<4, 2, uint16_t>(SLS_LZ_PASS_ARGS);
}

}  // namespace sls
