// Single-launch BiCGSTAB, F64 matrix values.
#include "persist.cuh"

namespace gko {

template <>
PkKernel<double, double> pk_bicg<double, double>(int shape, bool staged) {
  using T = double;
  using VT = double;
  GKO_PK_SHAPES(GKO_PK_BICG)
  GKO_PK_BLOCK_SHAPES(GKO_PK_BICG)
  return nullptr;
}

}  // namespace gko
