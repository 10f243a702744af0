// Interface between the C ABI layer and the tcgen05 (5th-generation tensor core) kernels.
#pragma once

#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include "../../include/xconv.h"

namespace xconv {

struct TcSketchPlan {
  int swap;            // 0: MMA rows = probes, columns = samples; 1: rows = samples, columns = probes
  int tile_m, tile_n, m_sub;  // output tile of one work unit; m_sub 128-row MMA tiles share the other operand
  int tiles_m, tiles_n, splits;
  bool row_boxes;            // operands are copied in boxes of eight rows x kgroup blocks
  int kgroup, rows_box;      // 64-wide k-blocks per stage; rows of the A box
  long kblocks, kblocks_per_split, kb_rem;   // the first kb_rem splits take one k-block more
  int stages;
  size_t part_bytes;
};

struct TcWgradPlan {
  // back-probe
  int bp_tile_n, bp_m_sub, bp_acc_bufs, bp_tiles_q, bp_tiles_r, bp_stages, bp_ksteps, bp_rows_box, bp_slots;
  int bp_groups;             // epilogue warps per tensor-memory lane quadrant
  long bp_base, bp_rem;      // column tiles: bp_base blocks of 64 positions each, the first bp_rem one more
  // contraction
  int ct_cw, ct_tile_n, ct_m_sub, ct_tiles_m, ct_tiles_n, ct_splits, ct_stages;
  int ct_tpu;                // kernel offsets per work unit (they share the L tile of every stage)
  int ct_halves;             // k-blocks copied and released in two halves; ct_stages then counts half-slots
  int ct_masked;             // block-sparse probes whose zero blocks are named: the contraction walks a list of the
                             // probes with a non-zero block per column tile (ct_list_bytes at the end of the partials)
  size_t ct_list_bytes;
  int patch_h, patch_w, patches_y, patches_x;
  long ct_items, ct_items_per_split, ct_items_rem;   // the first ct_items_rem splits take one item more
  size_t part_bytes;
};

struct TcConvPlan {
  int patch_w, patch_h;      // output pixels of one 128-row MMA tile
  int tile_n, tiles_n;       // channels out per column tile
  int m_sub, acc_bufs;       // patches that share each weight tile; accumulator sets in tensor memory
  int cw, nbw, ocw;          // channels per input tile row, per MN-major weight block (dX), per staging tile
  int resident, w_slots, a_slots;   // all weights in shared memory, or a ring of w_slots tiles; input boxes
  int o_per;                 // staging tiles per group of epilogue warps
  uint32_t a_sub_bytes;      // shared memory of one patch's box
  int groups;                // of epilogue warps: two where a patch is over quickly, one beside long mainloops, whose issue
                             // slots the second would only take
  long patches;
  int slide, ring;           // walk along an axis (conv_slide.cuh), patches then counts outputs; accumulators in the ring
};

struct TcHaloPlan {            // contraction of layers with few channels (contract_tc.cu)
  int pw, ph, stages;         // patch; stages of the ring
  int cwa, cwb;               // channels per block of L and of Z
  int rows_on_a;              // L moved by image rows on the MMA rows, else one dy per work unit
  int mt, mg_n, dy_n, dz_n, dz_per, ng_n, ng_per, j_n, j_per, a_blocks, cols;
  int drain;                  // accumulators added up in registers every few k-steps
  uint32_t a_blk, b_blk;      // shared memory of a channel block
  long patches, splits, units;
  size_t part_bytes;
};

struct StreamSketchPlan {      // sketch with at most 16 samples or 16 probes (stream_tc.cu)
  int swap;                   // 0: MMA rows = probes, columns = samples; 1: rows = samples
  int mt, nt, tiles_m, splits;
  size_t part_bytes;          // [split][r][B] float
};

// Fill the plan and say whether the tcgen05 kernels cover this layer.  tc_plan_wgrad returns a mask:
// bit 0 = back-probe covered, bit 1 = contraction covered.
bool tc_plan_sketch(const xconv_desc* d, TcSketchPlan* p, bool redraw = false);   // redraw: plan for a seeded call
int tc_plan_wgrad(const xconv_desc* d, TcWgradPlan* p);

bool tc_plan_conv(const xconv_desc* d, bool dgrad, TcConvPlan* p);
xconv_status tc_run_conv(const xconv_desc* d, const TcConvPlan& p, bool dgrad, const void* in, const void* W,
                         void* out, char* ws_head, cudaStream_t st);

// `seed` != nullptr: Z is not read; its tiles are redrawn inside the kernel from the Philox stream of *seed
// (Rademacher entries; see xconv_probes_from_seed).  Only for layers tc_sketch_can_redraw accepts.
xconv_status tc_run_sketch(const xconv_desc* d, const TcSketchPlan& p, const void* X, const void* Z, float* S,
                           char* ws_head, char* part, cudaStream_t st, const unsigned long long* seed = nullptr);
bool tc_sketch_can_redraw(const xconv_desc* d);
// `seed` != nullptr: the streamed operand (`dY`) is a set of probing vectors that is not read but redrawn inside
// the kernel from the Philox stream of *seed -- the first step of the estimator when it sums over the probes first.
xconv_status tc_run_backprobe(const xconv_desc* d, const TcWgradPlan& p, const void* S_bf16, const void* dY,
                              void* L, char* ws_head, cudaStream_t st, const unsigned long long* seed = nullptr);
bool tc_backprobe_row_boxes(const xconv_desc* d, bool seeded);      // dY copied eight rows at a time
xconv_status tc_run_contract(const xconv_desc* d, const TcWgradPlan& p, const void* L, const void* Z, float* dW,
                             float alpha, char* ws_head, char* part, cudaStream_t st);

bool tc_plan_halo(const xconv_desc* d, bool drain, TcHaloPlan* p);
// `cout_out`, `cin_out`: the channels of dW where d->Cout and d->Cin count padded ones.
xconv_status tc_run_halo(const xconv_desc* d, const TcHaloPlan& p, const void* L, const void* Z, int cout_out, int cin_out, float* dW,
                         float alpha, char* ws_head, char* part, cudaStream_t st);

// The streaming kernels for few samples or few probes.  The sketch leaves its partial sums in `part`; the back-probe takes
// S(row, k) = S[row * s_row + k * s_k], rows = d->r, reduction = d->B, and redraws its streamed operand if `seed` is given
// (H*W*Cout a multiple of 64 then).
bool tc_plan_sketch_stream(const xconv_desc* d, bool seeded, StreamSketchPlan* p);
xconv_status tc_run_sketch_stream(const xconv_desc* d, const StreamSketchPlan& p, const void* X, const void* Z, float* part,
                                  char* ws_head, cudaStream_t st, const unsigned long long* seed);
bool tc_backprobe_streams(const xconv_desc* d, bool other);
bool tc_stream_draws_pairs(const xconv_desc* d);                     // a warp of the seeded one takes two groups of 64 columns
// (`split`: S with more than its 16-bit rounding, see the kernel.)
xconv_status tc_run_backprobe_stream(const xconv_desc* d, const float* S, long s_row, long s_k, const void* dY, void* L,
                                     bool split, char* ws_head, cudaStream_t st, const unsigned long long* seed);

xconv_status tc_run_wait_selftest(char* ws_head, unsigned long long limit_ns, cudaStream_t st);

// bookkeeping shared with the ABI layer
void count_launch();
void set_cuda_error(int e);
unsigned int call_tag();   // tag of the API call in progress on this host thread

}  // namespace xconv
