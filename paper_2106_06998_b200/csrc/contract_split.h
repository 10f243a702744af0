// Offset contraction of float layers on the tensor cores (contract_split.cu).
#pragma once

#include "tc_api.h"

namespace xconv {

struct ContractSplitPlan {
  int rows_on_a, tiles, mg_n, dy_n, ng_n, j_n, j_per, ng_per, cols;   // work units (see the kernel's parameters)
  int cwa, a_blocks;            // channels per block of L, blocks
  int pw, ph, ksteps, stages, f_slots;
  uint32_t a_blk, b_blk, f_slot, f_b;
  long patches, splits, units;
  size_t part_bytes, bytes;     // partial sums; all scratch (with padded copies of L and Z)
};

bool plan_contract_split(const xconv_desc* d, ContractSplitPlan* p);
xconv_status run_contract_split(const xconv_desc* d, const ContractSplitPlan& p, const float* L, const float* Z, float* dW, float alpha,
                                char* ws_head, char* part, cudaStream_t st);

}  // namespace xconv
