// Single-launch CG, F64 matrix values.
#include "persist.cuh"

namespace gko {

template <>
PkKernel<double, double> pk_cg<double, double>(int shape, bool staged) {
  using T = double;
  using VT = double;
  GKO_PK_SHAPES(GKO_PK_CG)
  GKO_PK_BLOCK_SHAPES(GKO_PK_CG)
  return nullptr;
}

}  // namespace gko
