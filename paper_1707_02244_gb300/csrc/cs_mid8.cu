// Mid pass, radix-8 tiles of 64- to 1024-point rows.
#include "cs_col8.h"
#include "cs_mid.cuh"

namespace csk {

#define CS_SET_MID(k, T, S) \
  if (e == cudaSuccess) e = set_smem(mid_kernel<k, T, S>, T, 0, mid_smem_mult(k));
#define CS_L_MID(k, T, S) \
  case k: return launch_k(mid_kernel<k, T, S>, g.mid_ctas, T, VPT8, kp, s, mid_smem_mult(k));

cudaError_t mid8_init(const Geo& g) {
  cudaError_t e = cudaSuccess;
  switch (g.lgN1 + (g.twod ? 30 : 10)) {
    case 16: CS_MID_KINDS(CS_SET_MID, 256, 16) return e;
    case 17: CS_MID_KINDS(CS_SET_MID, 256, 17) return e;
    case 18: CS_MID_KINDS(CS_SET_MID, 512, 18) return e;
    case 19: CS_MID_KINDS(CS_SET_MID, 1024, 19) return e;
    case 20: CS_MID_KINDS(CS_SET_MID, 2048, 20) return e;
    case 36: CS_MID_KINDS_2D(CS_SET_MID, 256, 36) return e;
    case 37: CS_MID_KINDS_2D(CS_SET_MID, 256, 37) return e;
    case 38: CS_MID_KINDS_2D(CS_SET_MID, 512, 38) return e;
    case 39: CS_MID_KINDS_2D(CS_SET_MID, 1024, 39) return e;
    case 40: CS_MID_KINDS_2D(CS_SET_MID, 2048, 40) return e;
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t mid8_launch(MidKind kind, const KParams& kp, cudaStream_t s) {
  const Geo& g = kp.geo;
  switch (g.lgN1 + (g.twod ? 30 : 10)) {
    case 16: switch (kind) { CS_MID_KINDS(CS_L_MID, 256, 16) } break;
    case 17: switch (kind) { CS_MID_KINDS(CS_L_MID, 256, 17) } break;
    case 18: switch (kind) { CS_MID_KINDS(CS_L_MID, 512, 18) } break;
    case 19: switch (kind) { CS_MID_KINDS(CS_L_MID, 1024, 19) } break;
    case 20: switch (kind) { CS_MID_KINDS(CS_L_MID, 2048, 20) } break;
    case 36: switch (kind) { CS_MID_KINDS_2D(CS_L_MID, 256, 36) default: break; } break;
    case 37: switch (kind) { CS_MID_KINDS_2D(CS_L_MID, 256, 37) default: break; } break;
    case 38: switch (kind) { CS_MID_KINDS_2D(CS_L_MID, 512, 38) default: break; } break;
    case 39: switch (kind) { CS_MID_KINDS_2D(CS_L_MID, 1024, 39) default: break; } break;
    case 40: switch (kind) { CS_MID_KINDS_2D(CS_L_MID, 2048, 40) default: break; } break;
  }
  return cudaErrorInvalidValue;
}

}  // namespace csk
