// Single-launch GMRES, F64 matrix values.
#include "persist_gmres.cuh"

namespace gko {

template <>
PkGmresKernel<double, double> pk_gmres<double, double>(int shape, bool staged) {
  using T = double;
  using VT = double;
  GKO_PK_BLOCK_SHAPES(GKO_PK_GMRES)
  GKO_PK_GMRES(9, 512, 2, kPkGrid)
  GKO_PK_GMRES(10, 512, 4, kPkGrid)
  return nullptr;
}

}  // namespace gko
