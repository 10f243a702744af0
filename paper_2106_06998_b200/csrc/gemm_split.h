// Sketch and back-probe of float layers, and back-probe of 16-bit layers with S in parts, on the tensor cores (gemm_split.cu).
#pragma once

#include "tc_api.h"

namespace xconv {

struct GemmSplitPlan {
  int swap;                     // sketch: rows = samples (else probes)
  int n, tiles_n;               // columns per tile, tiles
  int stages, f_slots;          // of the ring of split tiles, of floats
  int f_rows_a, f_rows_b;       // rows of the boxes of floats
  long tiles_m, splits, kblocks;
  long clocks;                  // what the busiest SM is expected to take
  size_t bytes;                 // partial sums [split][r][B], or the split S
};

bool plan_sketch_split(const xconv_desc* d, GemmSplitPlan* p);
xconv_status run_sketch_split(const xconv_desc* d, const GemmSplitPlan& p, const float* X, const float* Z, float* part, char* ws_head,
                              cudaStream_t st);
// L[row][q] = sum over k of S[row * s_row + k * s_k] Y[k][q]: d->r rows, d->B terms.
bool plan_backprobe_split(const xconv_desc* d, GemmSplitPlan* p);
xconv_status run_backprobe_split(const xconv_desc* d, const GemmSplitPlan& p, const float* S, long s_row, long s_k, const void* Y, void* L,
                                 char* ws_head, char* scratch, cudaStream_t st);

}  // namespace xconv
