// Shared by the attention kernels and the insertion (Sec. 4.1, the attention half of delayed caching): argument block and
// the test for "this row is computed".
#pragma once

#include "team_common.cuh"

namespace team {

constexpr int kAttnMaxSplits = 8;      // portable cluster size

struct AttnArgs {
  const __nv_bfloat16* q;        // [T, Hq, d]
  const __nv_bfloat16* k_new;    // [T, Hkv, d]
  const __nv_bfloat16* v_new;
  const __nv_bfloat16* k_prefix; // [S, P, Hkv, d]
  const __nv_bfloat16* v_prefix;
  const int32_t* prefix_len;     // [S]
  __nv_bfloat16* k_block;        // [S, L, Hkv, d]
  __nv_bfloat16* v_block;
  const uint8_t* tok_state;      // [T]
  const int32_t* pos;
  const int32_t* group;
  const int32_t* branch;
  float* out;                    // [T, Hq, d]
  int32_t* status;               // [2] optional
  int S, B, L, Hq, Hkv, d, P, flags;
  int insert;                    // the attention kernel performs the insertion
};

__device__ __forceinline__ bool attn_computed(int state, int flags) { return !((flags & TEAM_F_DCD) && state == TEAM_TOK_CACHED); }

// the attention itself, on one of the kernels, with the insertion where *inserted comes back true; one-time set-up on a
// device's first call (team_attn_tc.cu)
cudaError_t launch_attention_tc(const AttnArgs& a, cudaStream_t s, bool* inserted);

// head size 64 on warp-level fragments (team_attn_frag.cu)
cudaError_t configure_attention_frag();
cudaError_t launch_attention_frag(const AttnArgs& a, int m_tiles, int n_splits, cudaStream_t s);

}  // namespace team
