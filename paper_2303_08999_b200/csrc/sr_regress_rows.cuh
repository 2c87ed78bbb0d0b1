// Regression of binary16 coefficients whose rows the tensor-core layouts cannot copy (any width, any alignment):
// declarations.
#pragma once
#include "sr_common.cuh"

namespace sr {

// Whether the call has the form that launch_regress_rows takes: dense or global subset, binary16 coefficients, atoms of 3 x 3,
// 5 x 5 or 7 x 7, up to four channels.
bool regress_rows_form(int mode, int coef_dtype, const Problem& pb);

// Whether a call of that form fits it and is expected to be faster there than on the thread-per-pixel kernel.
bool regress_rows_pay(int mode, const Problem& pb);

// The expected time of the faster of the two, us.
float regress_rows_or_general_us(int mode, const Problem& pb);

cudaError_t launch_regress_rows(int mode, const float* lr, const void* coef, const uint8_t* idx, const float* gamma, const float* dict,
                                float* out, const Problem& pb, cudaStream_t st);

} // namespace sr
