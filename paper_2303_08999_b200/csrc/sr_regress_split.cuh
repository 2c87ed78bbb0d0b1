// Small frames with every pixel's atoms dealt over several warps (sr_regress_split.cu).
#pragma once

#include "sr_common.cuh"

namespace sr {

// Whether the kernel takes a call: dense or global subset, 3 x 3 to 9 x 9 atoms, up to four channels, where one block for each
// multiprocessor covers the frames and there are atoms enough to deal out.
bool regress_split_pays(int mode, int coef_dtype, const Problem& pb);

cudaError_t launch_regress_split(int mode, const float* lr, const void* coef, int coef_dtype, const uint8_t* idx, const float* gamma,
                                 const float* dict, float* out, const Problem& pb, cudaStream_t st);

} // namespace sr
