// Single-launch GMRES, F32 matrix values.
#include "persist_gmres.cuh"

namespace gko {

template <>
PkGmresKernel<float, float> pk_gmres<float, float>(int shape, bool staged) {
  using T = float;
  using VT = float;
  GKO_PK_BLOCK_SHAPES(GKO_PK_GMRES)
  GKO_PK_GMRES(9, 512, 2, kPkGrid)
  GKO_PK_GMRES(10, 512, 4, kPkGrid)
  return nullptr;
}

}  // namespace gko
