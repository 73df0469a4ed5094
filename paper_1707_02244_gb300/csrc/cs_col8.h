// Radix-8 shapes of the passes (cs_col8a.cu, cs_col8b.cu, cs_mid8.cu).
#pragma once

#include "cs_internal.h"

namespace csk {

cudaError_t col8_init(const Geo& g);
cudaError_t col8_launch(ColKind kind, const KParams& kp, cudaStream_t s);
cudaError_t col8b_init(const Geo& g);
cudaError_t col8b_launch(ColKind kind, const KParams& kp, cudaStream_t s);
cudaError_t mid8_init(const Geo& g);
cudaError_t mid8_launch(MidKind kind, const KParams& kp, cudaStream_t s);

}  // namespace csk
