// Column pass: launchers, the run-time and the large static shapes.
#include "cs_col.cuh"
#include "cs_col8.h"

namespace csk {

cudaError_t init_col_kernels(const Geo& g) {
  if (g.col_r8) return col8_init(g);
  cudaError_t e = cudaSuccess;
#define CS_SET_COL(k, S) \
  if (e == cudaSuccess) e = set_smem(col_kernel<k, S>, ColTile<S>::kTile, ColTile<S>::kMinB);
  if (g.col_tile == COL_TILE4) {
    CS_COL_KINDS_2D(CS_SET_COL, 3)
  } else if (g.col_tile == COL_TILE2) {
    CS_COL_KINDS_2D(CS_SET_COL, 5)
  } else if (g.lgN2 == 10 && g.lgG == 2) {
    CS_COL_KINDS(CS_SET_COL, 1)
  } else {
    CS_COL_KINDS(CS_SET_COL, 0)
  }
#undef CS_SET_COL
  return e;
}

cudaError_t launch_col(ColKind kind, const KParams& kp, cudaStream_t s) {
  const Geo& g = kp.geo;
  const int grid = g.col_ctas;
  const bool hot = g.lgN2 == 10 && g.lgG == 2;
  if (g.col_r8) return col8_launch(kind, kp, s);
#define CS_L_COL(k, S) case k: return launch_k(col_kernel<k, S>, grid, ColTile<S>::kTile, EPT, kp, s);
  if (g.col_tile == COL_TILE4) {
    if (g.lgN2 == 12 && g.lgG == 2) {
      switch (kind) { CS_COL_KINDS_2D(CS_L_COL, 3) default: break; }
    }
  } else if (g.col_tile == COL_TILE2) {
    if (g.lgN2 == 11 && g.lgG == 2) {
      switch (kind) { CS_COL_KINDS_2D(CS_L_COL, 5) default: break; }
    }
  } else if (hot) {
    switch (kind) { CS_COL_KINDS(CS_L_COL, 1) }
  } else {
    switch (kind) { CS_COL_KINDS(CS_L_COL, 0) }
  }
#undef CS_L_COL
  return cudaErrorInvalidValue;
}

}  // namespace csk
