// Direct convolution on FP32 multiply-adds for float storage (conv_fma.cu).
#pragma once

#include "tc_api.h"

namespace xconv {

// Block and patch of a launch; plane: floats of one input channel in shared memory.
struct ConvFma { int threads, tn, SW, RH, NI, pitch, plane; };

bool plan_conv_fma(const xconv_desc* d, bool dgrad, ConvFma* g);
xconv_status run_conv_fma(const xconv_desc* d, const ConvFma& g, bool dgrad, const float* in, const float* Wt, float* out,
                          cudaStream_t st);

}  // namespace xconv
