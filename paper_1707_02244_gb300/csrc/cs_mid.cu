// Mid pass: launchers, the run-time and the large static shapes, and the
// grouped launches of the batched solves.
#include "cs_col8.h"
#include "cs_mid.cuh"

namespace csk {

namespace {

// Grouped launch over many plans (batched solves): CTA b runs tile
// map[b].y of plan map[b].x (4096-value tiles, run-time shapes).
template <int KIND>
__global__ void __launch_bounds__(Cfg<4096>::NT, Cfg<4096>::MINB)
    mid_kernel_multi(const KParams* __restrict__ kps, const int2* __restrict__ map) {
  static_assert(sizeof(KParams) % 4 == 0 && sizeof(KParams) / 4 <= Cfg<4096>::NT, "KParams copy");
  __shared__ KParams skp;
  const int2 it = map[blockIdx.x];
  if (threadIdx.x < sizeof(KParams) / 4)
    reinterpret_cast<int*>(&skp)[threadIdx.x] = reinterpret_cast<const int*>(kps + it.x)[threadIdx.x];
  __syncthreads();
  mid_body<KIND, 4096, 0>(skp, it.y);
}

}  // namespace

// The static shape that geometry g launches, or 0 / 4 (run-time shapes).
static int mid_shape(const Geo& g) {
  if (g.twod) {
    if (g.lgN1 == 11 && g.lgU == 0 && g.tile == 4096) return 5;
    if (g.lgN1 == 12 && g.lgU == 0 && g.tile == 8192) return 6;
    return 4;
  }
  if (g.lgN1 == 10 && g.lgU == 1 && g.tile == 4096) return 1;
  if (g.lgN1 == 11 && g.lgU == 0 && g.tile == 4096) return 2;
  if (g.lgN1 == 12 && g.lgU == 0 && g.tile == 8192) return 3;
  return 0;
}

cudaError_t init_mid_kernels(const Geo& g) {
  if (g.mid_r8) return mid8_init(g);
  cudaError_t e = cudaSuccess;
#define CS_SET_MID(k, T, S) \
  if (e == cudaSuccess) e = set_smem(mid_kernel<k, T, S>, T, Cfg<T>::MINB, mid_smem_mult(k));
  switch (mid_shape(g)) {
    case 1: CS_MID_KINDS(CS_SET_MID, 4096, 1) break;
    case 2: CS_MID_KINDS(CS_SET_MID, 4096, 2) break;
    case 3: CS_MID_KINDS(CS_SET_MID, 8192, 3) break;
    case 5: CS_MID_KINDS_2D(CS_SET_MID, 4096, 5) break;
    case 6: CS_MID_KINDS_2D(CS_SET_MID, 8192, 6) break;
    case 4:
      if (g.tile == 4096) { CS_MID_KINDS_2D(CS_SET_MID, 4096, 4) }
      else { CS_MID_KINDS_2D(CS_SET_MID, 8192, 4) }
      break;
    default:
      if (g.tile == 4096) { CS_MID_KINDS(CS_SET_MID, 4096, 0) }
      else { CS_MID_KINDS(CS_SET_MID, 8192, 0) }
  }
#undef CS_SET_MID
  return e;
}

cudaError_t launch_mid(MidKind kind, const KParams& kp, cudaStream_t s) {
  const Geo& g = kp.geo;
  if (g.mid_r8) return mid8_launch(kind, kp, s);
  const int grid = g.mid_ctas;
#define CS_L_MID(k, T, S) case k: return launch_k(mid_kernel<k, T, S>, grid, T, EPT, kp, s, mid_smem_mult(k));
  switch (mid_shape(g)) {
    case 1: switch (kind) { CS_MID_KINDS(CS_L_MID, 4096, 1) } break;
    case 2: switch (kind) { CS_MID_KINDS(CS_L_MID, 4096, 2) } break;
    case 3: switch (kind) { CS_MID_KINDS(CS_L_MID, 8192, 3) } break;
    case 5: switch (kind) { CS_MID_KINDS_2D(CS_L_MID, 4096, 5) default: break; } break;
    case 6: switch (kind) { CS_MID_KINDS_2D(CS_L_MID, 8192, 6) default: break; } break;
    case 4:
      if (g.tile == 4096) { switch (kind) { CS_MID_KINDS_2D(CS_L_MID, 4096, 4) default: break; } }
      else { switch (kind) { CS_MID_KINDS_2D(CS_L_MID, 8192, 4) default: break; } }
      break;
    default:
      if (g.tile == 4096) { switch (kind) { CS_MID_KINDS(CS_L_MID, 4096, 0) } }
      else { switch (kind) { CS_MID_KINDS(CS_L_MID, 8192, 0) } }
  }
#undef CS_L_MID
  return cudaErrorInvalidValue;
}

#define CS_MID_KINDS_MULTI(X) X(MID_FWD) X(MID_ADJ) X(MID_ADMM)

cudaError_t init_mid_multi_kernels() {
  cudaError_t e = cudaSuccess;
#define CS_SET_MIDM(k) \
  if (e == cudaSuccess) e = set_smem(mid_kernel_multi<k>, 4096, Cfg<4096>::MINB);
  CS_MID_KINDS_MULTI(CS_SET_MIDM)
#undef CS_SET_MIDM
  return e;
}

cudaError_t launch_mid_multi(MidKind kind, const KParams* kps, const int2* map, int nctas, cudaStream_t s) {
  if (nctas < 1) return cudaSuccess;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(nctas);
  cfg.blockDim = dim3(Cfg<4096>::NT);
  cfg.dynamicSmemBytes = pass_smem_bytes(4096);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  switch (kind) {
    case MID_FWD: return cudaLaunchKernelEx(&cfg, mid_kernel_multi<MID_FWD>, kps, map);
    case MID_ADJ: return cudaLaunchKernelEx(&cfg, mid_kernel_multi<MID_ADJ>, kps, map);
    case MID_ADMM: return cudaLaunchKernelEx(&cfg, mid_kernel_multi<MID_ADMM>, kps, map);
    default: break;
  }
  return cudaErrorInvalidValue;
}

size_t pass_smem_bytes(int tile) { return sizeof(float2) * (size_t)smem_slots(tile); }

}  // namespace csk
