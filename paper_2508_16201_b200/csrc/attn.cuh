// Parameters shared by the attention kernels and their launchers.
#pragma once
#include "common.cuh"

namespace specvlm {

struct AttnParams {
  const __nv_bfloat16* q;     // [L][B][n_q][Hq][D]
  __nv_bfloat16* out;         // same shape
  float* lse;                 // [L][B][n_q][Hq] or null
  const int32_t* block_table; // [B][max_blocks] or null
  const int32_t* seq_lens;    // [B]
  int32_t* d_status;
  int32_t batch, n_q, n_q_heads, n_kv_heads, group, rows;   // rows = group * n_q
  int32_t max_blocks, block_tokens, max_seq_len;
  float scale_log2;           // sm_scale * log2(e)
  int32_t lost_cta;           // test hook: the CTA that gives up as if a wait had expired; -1 as a rule
};

}  // namespace specvlm
