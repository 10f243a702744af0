// Convolution and offset contraction of small float layers (small_f32.cu).
#pragma once

#include <cuda_runtime.h>

#include "../../include/xconv.h"

namespace xconv {

// The convolution (the input gradient with `dgrad`) of a small float layer whose channel counts are multiples of 4, without circular shifts.
bool small_conv_serves(const xconv_desc* d);
xconv_status run_small_conv(const xconv_desc* d, bool dgrad, const float* in, const float* Wt, float* out, cudaStream_t st);

// The contraction of channel counts that are multiples of 4 and leave most of the 32 x 64 channels of contract_simt_async empty, in its split of the work items
// (probe, row, 32 pixels): partial sums [split][Cout][offsets][Cin].
bool small_contract_serves(const xconv_desc* d);
xconv_status run_small_contract(const xconv_desc* d, int splits, long items_per_split, const float* L, const float* Z, float* part, cudaStream_t st);

}  // namespace xconv
