// What a step from host buffers and one on device buffers share.
#pragma once
#include "common.cuh"

namespace ss {
namespace attn {
// ss_tree_attention.  `q_ready` (may be null): an event that the stream waits for in front of the first kernel that reads the
// queries, which is not the planner.  `out_on_host`: the rows go over the bus as they are written.
int32_t tree_attention(const ss_attn_desc_t* d, void* workspace, size_t workspace_bytes, void* stream, cudaEvent_t q_ready,
                       bool out_on_host);
}  // namespace attn
// ss_candidate_step, likewise.
int32_t candidate_step(const ss_device_step_t& s, void* stream, cudaEvent_t q_ready, bool out_on_host);
}  // namespace ss
