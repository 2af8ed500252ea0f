// Single-launch BiCGSTAB, BF16 matrix values.
#include "persist.cuh"

namespace gko {

template <>
PkKernel<float, __nv_bfloat16> pk_bicg<float, __nv_bfloat16>(int shape, bool staged) {
  using T = float;
  using VT = __nv_bfloat16;
  GKO_PK_SHAPES(GKO_PK_BICG)
  GKO_PK_BLOCK_SHAPES(GKO_PK_BICG)
  return nullptr;
}

}  // namespace gko
