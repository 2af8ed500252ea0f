// Single-launch CG, BF16 matrix values.
#include "persist.cuh"

namespace gko {

template <>
PkKernel<float, __nv_bfloat16> pk_cg<float, __nv_bfloat16>(int shape, bool staged) {
  using T = float;
  using VT = __nv_bfloat16;
  GKO_PK_SHAPES(GKO_PK_CG)
  GKO_PK_BLOCK_SHAPES(GKO_PK_CG)
  return nullptr;
}

}  // namespace gko
