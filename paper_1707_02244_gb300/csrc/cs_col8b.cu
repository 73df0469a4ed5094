// Column pass, radix-8 tiles of 256- and 512-point columns.
#include "cs_col.cuh"
#include "cs_col8.h"

namespace csk {

#define CS_SET_COL(k, S) \
  if (e == cudaSuccess) e = set_smem(col_kernel<k, S>, ColTile<S>::kTile, ColTile<S>::kCarve);
#define CS_L_COL(k, S) case k: return launch_k(col_kernel<k, S>, g.col_ctas, ColTile<S>::kTile, VPT8, kp, s);

cudaError_t col8b_init(const Geo& g) {
  cudaError_t e = cudaSuccess;
  switch (g.lgN2) {
    case 8: CS_COL_KINDS(CS_SET_COL, 18) return e;
    case 9: CS_COL_KINDS(CS_SET_COL, 19) return e;
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t col8b_launch(ColKind kind, const KParams& kp, cudaStream_t s) {
  const Geo& g = kp.geo;
  switch (g.lgN2) {
    case 8: switch (kind) { CS_COL_KINDS(CS_L_COL, 18) } break;
    case 9: switch (kind) { CS_COL_KINDS(CS_L_COL, 19) } break;
    default: return cudaErrorInvalidValue;
  }
  return cudaErrorInvalidValue;
}

}  // namespace csk
