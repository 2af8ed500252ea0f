// Single-launch CG, F32 matrix values.
#include "persist.cuh"

namespace gko {

template <>
PkKernel<float, float> pk_cg<float, float>(int shape, bool staged) {
  using T = float;
  using VT = float;
  GKO_PK_SHAPES(GKO_PK_CG)
  GKO_PK_BLOCK_SHAPES(GKO_PK_CG)
  return nullptr;
}

}  // namespace gko
