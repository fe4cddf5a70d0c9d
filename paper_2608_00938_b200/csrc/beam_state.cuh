// Beam-state update after a selection (Sections 3.3, 4.4): the child's node and the extended prefix key of one chosen
// candidate.  Shared by the update kernel and by the selection that finishes with it.
#pragma once
#include "common.cuh"

namespace grace {

struct BeamUpdate {
  const int32_t* prev_node;
  const uint64_t* prev_key;
  const uint64_t* child_bits;
  const int32_t* child_base;
  int32_t* new_node;             // nullptr: no update asked for
  uint64_t* new_key;
  int64_t num_internal;
  int M_prev, V, prefix_len;
};

// Entry i of the new beam of request b was reached from parent `par` with token `tok` and score `score`.
__device__ __forceinline__ void beam_update_one(const BeamUpdate& u, int64_t i, int b, int par, int tok, float score,
                                                int32_t* d_status) {
  if (par < 0 || par >= u.M_prev || tok < 0 || tok >= u.V) {
    flag_status(d_status, GRACE_DEV_BAD_INDEX);
    u.new_node[i] = -1;
    u.new_key[i] = 0;
    return;
  }
  const int64_t src = (int64_t)b * u.M_prev + par;
  u.new_key[i] = u.prev_key[src] | ((uint64_t)(tok + 1) << (16 * u.prefix_len));
  const int node = u.prev_node[src];
  int out = -1;
  if (node >= 0 && node < u.num_internal && score != __int_as_float(0xff800000)) {
    const uint64_t* row = u.child_bits + (int64_t)node * (u.V >> 6);
    const uint64_t word = __ldg(row + (tok >> 6));
    const int base = __ldg(u.child_base + node);
    if ((word >> (tok & 63)) & 1ull) {
      int rank = __popcll(word & ((1ull << (tok & 63)) - 1ull));
#pragma unroll 8
      for (int w = 0; w < (tok >> 6); ++w) rank += __popcll(__ldg(row + w));
      out = base + rank;
    }
  }
  u.new_node[i] = out;
}

}  // namespace grace
