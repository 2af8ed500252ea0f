// Single-launch GMRES, BF16 matrix values.
#include "persist_gmres.cuh"

namespace gko {

template <>
PkGmresKernel<float, __nv_bfloat16> pk_gmres<float, __nv_bfloat16>(int shape, bool staged) {
  using T = float;
  using VT = __nv_bfloat16;
  GKO_PK_BLOCK_SHAPES(GKO_PK_GMRES)
  GKO_PK_GMRES(9, 512, 2, kPkGrid)
  GKO_PK_GMRES(10, 512, 4, kPkGrid)
  return nullptr;
}

}  // namespace gko
