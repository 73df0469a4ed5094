// Grouped launches of the batched solves: one pass over the tiles of every
// plan of one length, 4096-value tiles with the shape fixed at compile time.
#include "cs_col.cuh"
#include "cs_mid.cuh"

namespace csk {

namespace {

// CTA b runs tile map[b].y of plan map[b].x, whose parameters kps[map[b].x]
// are copied to shared memory first.
template <int NT>
__device__ __forceinline__ int fetch_plan(KParams& skp, const KParams* __restrict__ kps, const int2* __restrict__ map) {
  static_assert(sizeof(KParams) % 4 == 0 && sizeof(KParams) / 4 <= NT, "KParams copy");
  const int2 it = map[blockIdx.x];
  if (threadIdx.x < sizeof(KParams) / 4)
    reinterpret_cast<int*>(&skp)[threadIdx.x] = reinterpret_cast<const int*>(kps + it.x)[threadIdx.x];
  __syncthreads();
  return it.y;
}

template <int KIND, int SHAPE>
__global__ void __launch_bounds__(COL_TILE / EPT, COL_MINB)
    col_kernel_multi(const KParams* __restrict__ kps, const int2* __restrict__ map) {
  __shared__ KParams skp;
  const int blk = fetch_plan<COL_TILE / EPT>(skp, kps, map);
  col_body<KIND, SHAPE>(skp, blk);
}

template <int KIND, int SHAPE>
__global__ void __launch_bounds__(Cfg<4096>::NT, Cfg<4096>::MINB)
    mid_kernel_multi(const KParams* __restrict__ kps, const int2* __restrict__ map) {
  __shared__ KParams skp;
  const int blk = fetch_plan<Cfg<4096>::NT>(skp, kps, map);
  mid_body<KIND, 4096, SHAPE>(skp, blk);
}

template <typename K>
cudaError_t launch_multi(K kern, int grid, const KParams* kps, const int2* map, cudaStream_t s) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(4096 / EPT);
  cfg.dynamicSmemBytes = pass_smem_bytes(4096);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, kps, map);
}

// Lengths N = 2^13 .. 2^21: columns of 2^6 .. 2^10, rows of 2^7 .. 2^11.
#define CS_COL_KINDS_MULTI(X, S) \
  X(COL_LOAD, S) X(COL_RESIDUAL, S) X(COL_ISTA, S) X(COL_ISTA_LAST, S) X(COL_ADMM_INIT, S) X(COL_ADMM, S) \
  X(COL_ADMM_LAST, S)
#define CS_MID_KINDS_MULTI(X, S) X(MID_FWD, S) X(MID_ADJ, S) X(MID_ADMM, S)
#define CS_COL_SHAPES(X, K) X(6, K, 46) X(7, K, 47) X(8, K, 48) X(9, K, 49) X(10, K, 50)
#define CS_MID_SHAPES(X, K) X(7, K, 57) X(8, K, 58) X(9, K, 59) X(10, K, 60) X(11, K, 61)

bool multi_geo(const Geo& g) {
  return !g.twod && !g.col_r8 && !g.mid_r8 && g.tile == 4096 && g.col_tile == 4096 && g.lgN2 >= 6 && g.lgN2 <= 10 &&
         g.lgG == 12 - g.lgN2 && g.lgN1 >= 7 && g.lgN1 <= 11 && g.lgU == 11 - g.lgN1;
}

}  // namespace

cudaError_t init_multi_kernels(const Geo& g) {
  if (!multi_geo(g)) return cudaErrorInvalidValue;
  cudaError_t e = cudaSuccess;
#define CS_SET_COLM(k, S) if (e == cudaSuccess) e = set_smem(col_kernel_multi<k, S>, COL_TILE, COL_MINB);
#define CS_SET_MIDM(k, S) if (e == cudaSuccess) e = set_smem(mid_kernel_multi<k, S>, 4096, Cfg<4096>::MINB);
#define CS_CASE(l, K, S) case l: K(S) break;
#define CS_COLM(S) CS_COL_KINDS_MULTI(CS_SET_COLM, S)
#define CS_MIDM(S) CS_MID_KINDS_MULTI(CS_SET_MIDM, S)
  switch (g.lgN2) { CS_COL_SHAPES(CS_CASE, CS_COLM) }
  switch (g.lgN1) { CS_MID_SHAPES(CS_CASE, CS_MIDM) }
#undef CS_MIDM
#undef CS_COLM
#undef CS_SET_MIDM
#undef CS_SET_COLM
  return e;
}

cudaError_t launch_col_multi(ColKind kind, const Geo& g, const KParams* kps, const int2* map, int nctas,
                             cudaStream_t s) {
  if (nctas < 1) return cudaSuccess;
#define CS_L_COLM(k, S) case k: return launch_multi(col_kernel_multi<k, S>, nctas, kps, map, s);
#define CS_COLM(S) switch (kind) { CS_COL_KINDS_MULTI(CS_L_COLM, S) default: break; }
  switch (g.lgN2) { CS_COL_SHAPES(CS_CASE, CS_COLM) }
#undef CS_COLM
#undef CS_L_COLM
  return cudaErrorInvalidValue;
}

cudaError_t launch_mid_multi(MidKind kind, const Geo& g, const KParams* kps, const int2* map, int nctas,
                             cudaStream_t s) {
  if (nctas < 1) return cudaSuccess;
#define CS_L_MIDM(k, S) case k: return launch_multi(mid_kernel_multi<k, S>, nctas, kps, map, s);
#define CS_MIDM(S) switch (kind) { CS_MID_KINDS_MULTI(CS_L_MIDM, S) default: break; }
  switch (g.lgN1) { CS_MID_SHAPES(CS_CASE, CS_MIDM) }
#undef CS_MIDM
#undef CS_L_MIDM
#undef CS_CASE
  return cudaErrorInvalidValue;
}

}  // namespace csk
