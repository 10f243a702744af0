// Convolution of float layers on the tensor cores (conv_split.cu).
#pragma once

#include "tc_api.h"

namespace xconv {

struct ConvSplitPlan {
  int cw, nb, ks_last;          // channels in per block, blocks, k-steps of the last one
  int n, tiles_n, ocw;          // channels out per column tile, tiles, channels per staging tile
  int pw, ph;                   // patch
  long patches;
  uint32_t a_plane, w_tile, f_slot;
  int a_slots, w_slots, f_slots;
  size_t img_bytes, bytes;      // the split weights; all scratch behind the header (with a padded copy of the input)
};

// The padded copy of a float tensor whose rows are no multiple of 16 bytes (`t` is the copy then).
size_t padded_float_bytes(long rows, int C);
xconv_status pad_floats(const float*& t, float* copy, long rows, int C, cudaStream_t st);

bool plan_conv_split(const xconv_desc* d, bool dgrad, ConvSplitPlan* p);
xconv_status run_conv_split(const xconv_desc* d, const ConvSplitPlan& p, bool dgrad, const float* in, const float* Wt, float* out,
                            char* ws_head, char* scratch, cudaStream_t st);

}  // namespace xconv
