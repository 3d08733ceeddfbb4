// Internal declarations of the decoder library.
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>

namespace decoder {

constexpr int kPlain = 0, kResid = 1, kSwiglu = 2;

// cuTensorMapEncodeTiled, by the driver's entry point (NULL: none).
using EncodeFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                              const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                              CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
EncodeFn encode_fn();

// The current device's error word (see decoder_error).
unsigned* error_word();

// The fused projections of gemm.cu (see decoder_gemm) and the shapes they take.
bool gemm_takes(int M, int N, int K);
int gemm(int mode, const void* x, const void* w0, const void* w1, const void* h, void* y, int M, int N, int K,
         cudaStream_t stream);

}  // namespace decoder
