// Exact decode under independent X/Z noise at FP64 accuracy by the column
// transfer (mld_xz.cu).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "mld_internal.h"

namespace mld {

// Arguments as mld_decode_xz (checked, the code's device tables made);
// asynchronous on s after the first call for a code.
mld_status decode_xz_fp64(mld_code* C, const float* px, const float* pz, const uint64_t* syn, int64_t B, double* logP,
                          uint8_t* argmax, cudaStream_t s);
// Flops executed since the last call (then reset).
mld_status xz_fp64_flops(mld_code* C, double* flops);

}  // namespace mld
