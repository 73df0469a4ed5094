// Column pass: launchers, the run-time and the large static shapes, and the
// grouped launches of the batched solves.
#include "cs_col.cuh"
#include "cs_col8.h"

namespace csk {

namespace {

// Grouped launch over many plans (batched solves): CTA b runs tile
// map[b].y of plan map[b].x, whose parameters kps[map[b].x] are copied to
// shared memory first.  Run-time shapes only.
template <int KIND>
__global__ void __launch_bounds__(COL_TILE / EPT, COL_MINB)
    col_kernel_multi(const KParams* __restrict__ kps, const int2* __restrict__ map) {
  static_assert(sizeof(KParams) % 4 == 0 && sizeof(KParams) / 4 <= COL_TILE / EPT, "KParams copy");
  __shared__ KParams skp;
  const int2 it = map[blockIdx.x];
  if (threadIdx.x < sizeof(KParams) / 4)
    reinterpret_cast<int*>(&skp)[threadIdx.x] = reinterpret_cast<const int*>(kps + it.x)[threadIdx.x];
  __syncthreads();
  col_body<KIND, 0>(skp, it.y);
}

}  // namespace

cudaError_t init_col_kernels(const Geo& g) {
  if (g.col_r8) return col8_init(g);
  cudaError_t e = cudaSuccess;
#define CS_SET_COL(k, S) \
  if (e == cudaSuccess) e = set_smem(col_kernel<k, S>, ColTile<S>::kTile, ColTile<S>::kMinB);
  if (g.col_tile == COL_TILE4) {
    CS_COL_KINDS_2D(CS_SET_COL, 3)
  } else if (g.lgN2 == 10 && g.lgG == 2) {
    CS_COL_KINDS(CS_SET_COL, 1)
  } else {
    CS_COL_KINDS(CS_SET_COL, 0)
  }
#undef CS_SET_COL
  return e;
}

#define CS_COL_KINDS_MULTI(X) \
  X(COL_LOAD) X(COL_RESIDUAL) X(COL_ISTA) X(COL_ISTA_LAST) X(COL_ADMM_INIT) X(COL_ADMM) X(COL_ADMM_LAST)

cudaError_t init_col_multi_kernels() {
  cudaError_t e = cudaSuccess;
#define CS_SET_COLM(k) \
  if (e == cudaSuccess) e = set_smem(col_kernel_multi<k>, COL_TILE, COL_MINB);
  CS_COL_KINDS_MULTI(CS_SET_COLM)
#undef CS_SET_COLM
  return e;
}

template <typename K>
cudaError_t launch_multi(K kern, int grid, int tile, const KParams* kps, const int2* map, cudaStream_t s,
                         int smem_mult = 1) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(tile / EPT);
  cfg.dynamicSmemBytes = smem_mult * pass_smem_bytes(tile);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, kps, map);
}

cudaError_t launch_col_multi(ColKind kind, const KParams* kps, const int2* map, int nctas, cudaStream_t s) {
  if (nctas < 1) return cudaSuccess;
#define CS_L_COLM(k) case k: return launch_multi(col_kernel_multi<k>, nctas, COL_TILE, kps, map, s);
  switch (kind) {
    CS_COL_KINDS_MULTI(CS_L_COLM)
    default: break;
  }
#undef CS_L_COLM
  return cudaErrorInvalidValue;
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
  } else if (hot) {
    switch (kind) { CS_COL_KINDS(CS_L_COL, 1) }
  } else {
    switch (kind) { CS_COL_KINDS(CS_L_COL, 0) }
  }
#undef CS_L_COL
  return cudaErrorInvalidValue;
}

}  // namespace csk
