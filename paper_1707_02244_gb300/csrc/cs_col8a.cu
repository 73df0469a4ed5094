// Column pass, radix-8 tiles of 32- to 128-point columns.
#include "cs_col.cuh"
#include "cs_col8.h"

namespace csk {

#define CS_SET_COL(k, S) \
  if (e == cudaSuccess) e = set_smem(col_kernel<k, S>, ColTile<S>::kTile, ColTile<S>::kCarve);
#define CS_L_COL(k, S) case k: return launch_k(col_kernel<k, S>, g.col_ctas, ColTile<S>::kTile, VPT8, kp, s);

cudaError_t col8_init(const Geo& g) {
  cudaError_t e = cudaSuccess;
  switch (g.lgN2) {
    case 5: CS_COL_KINDS(CS_SET_COL, 15) return e;
    case 6: CS_COL_KINDS(CS_SET_COL, 16) return e;
    case 7: CS_COL_KINDS(CS_SET_COL, 17) return e;
    default: return col8b_init(g);
  }
}

cudaError_t col8_launch(ColKind kind, const KParams& kp, cudaStream_t s) {
  const Geo& g = kp.geo;
  switch (g.lgN2) {
    case 5: switch (kind) { CS_COL_KINDS(CS_L_COL, 15) } break;
    case 6: switch (kind) { CS_COL_KINDS(CS_L_COL, 16) } break;
    case 7: switch (kind) { CS_COL_KINDS(CS_L_COL, 17) } break;
    default: return col8b_launch(kind, kp, s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace csk
