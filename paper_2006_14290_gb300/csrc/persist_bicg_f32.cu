// Single-launch BiCGSTAB, F32 matrix values.
#include "persist.cuh"

namespace gko {

template <>
PkKernel<float, float> pk_bicg<float, float>(int shape, bool staged) {
  using T = float;
  using VT = float;
  GKO_PK_SHAPES(GKO_PK_BICG)
  GKO_PK_BLOCK_SHAPES(GKO_PK_BICG)
  return nullptr;
}

}  // namespace gko
