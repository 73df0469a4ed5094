// Mid pass: launchers, the run-time and the large static shapes.
#include "cs_col8.h"
#include "cs_mid.cuh"

namespace csk {

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

size_t pass_smem_bytes(int tile) { return sizeof(float2) * (size_t)smem_slots(tile); }

}  // namespace csk
