// Register-tiled regression on the fp32 FMA pipe (fp32 coefficients, dense and global-subset calls): declarations.
#pragma once
#include "sr_common.cuh"

namespace sr {

// Whether launch_regress_tile takes the call: dense or global subset, fp32 coefficients of any width and alignment, up to
// four channels, enough pixels to fill the chip.
bool regress_tile_supported(int mode, int coef_dtype, const Problem& pb);

cudaError_t launch_regress_tile(int mode, const float* lr, const void* coef, const uint8_t* idx, const float* gamma, const float* dict,
                                float* out, const Problem& pb, cudaStream_t st);

} // namespace sr
