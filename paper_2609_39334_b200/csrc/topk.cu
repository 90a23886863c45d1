// ss_topk_prune: keep the k best-scored candidates of every problem (paper, Section "Early Pruning of Search
// Tree": a candidate ranked below the top-k cannot be selected; Section "Test-Time Scaling": k = N / M).
//
// One block per segment.  Each candidate becomes a 64-bit key (order-reversed score bits << 32 | local
// index), so ascending key order is "score descending, index ascending" and all keys are distinct.  A segment of up to one
// candidate per thread is sorted in registers (a bitonic network, partners in the warp through shuffles, the others through
// shared memory), a larger one in shared memory (up to kSmemKeys) or in the caller's workspace; then the first k indices
// and the mask are written.
// Latency-bound.  One launch and nothing else: block 0 checks all segments, writes the status word and clears the mask
// outside every segment.  Measured, in the kernel: 64 segments of 256 half verified 4.6 us, 16 segments of 64 3.0, 4 of 256 3.8; the
// early pruning call 16.4 -> 6.2 us (two memsets in front of a shared-memory network with a barrier per stage before).
#include "topk.cuh"

namespace ss {
namespace topk {

__global__ void __launch_bounds__(kMaxThreads)
topk_kernel(const float* __restrict__ scores, const int32_t* __restrict__ seg_offsets, int n_total, int k,
            int32_t* __restrict__ survivors, uint8_t* __restrict__ keep, uint64_t* __restrict__ scratch,
            int32_t* __restrict__ status) {
  ss::grid_dependency_enter();
  __shared__ uint64_t smem_keys[kSmemKeys];
  select_segment(blockIdx.x, gridDim.x, scores, seg_offsets, n_total, k, survivors, keep, scratch, status, smem_keys);
}

// Early pruning with partially verified candidates (paper, Section "Early Pruning of Search Tree").  Same sort as
// above over the VERIFIED candidates only (the others get keys that sort last); then
//   rule 2: >= k verified candidates with the perfect score  -> the first k of them by index are selected, every
//           other candidate of the segment is pruned, the segment is final;
//   rule 1: more than k verified -> the verified candidates ranked below the k best are pruned;
//   all verified -> final, selected = the k best.
__device__ __forceinline__ void early_prune_segment(const float* __restrict__ scores, const uint8_t* __restrict__ verified,
                                                    const Segment g, int k, uint8_t* __restrict__ pruned,
                                                    int32_t* __restrict__ selected, uint8_t* __restrict__ final_out,
                                                    uint64_t* __restrict__ scratch, uint64_t* smem_keys, int& s_nver, int& s_nperfect) {
  __shared__ int s_warp[32];
  const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, warp = tid >> 5;
  int32_t* out = selected + static_cast<int64_t>(blockIdx.x) * k;
  if (g.n == 0) {
    for (int j = tid; j < k; j += nt) out[j] = -1;
    if (tid == 0) final_out[blockIdx.x] = 1;      // nothing left to verify in an empty segment
    return;
  }
  __syncthreads();
  int my_ver = 0, my_perfect = 0;
  for (int i = tid; i < g.n; i += nt) {
    if (!verified[g.lo + i]) continue;
    ++my_ver;
    if (scores[g.lo + i] >= 1.0f) ++my_perfect;
  }
  my_ver = static_cast<int>(__reduce_add_sync(0xffffffffu, static_cast<unsigned>(my_ver)));
  my_perfect = static_cast<int>(__reduce_add_sync(0xffffffffu, static_cast<unsigned>(my_perfect)));
  if (lane == 0 && my_ver) atomicAdd(&s_nver, my_ver);
  if (lane == 0 && my_perfect) atomicAdd(&s_nperfect, my_perfect);
  __syncthreads();
  const int nver = s_nver, nperfect = s_nperfect;
  if (nperfect >= k) {                            // rule 2: rank of a perfect candidate among the perfect ones by index
    int before = 0;
    for (int base = 0; base < g.n; base += nt) {
      const int i = base + tid;
      const bool perfect = i < g.n && verified[g.lo + i] && scores[g.lo + i] >= 1.0f;
      const uint32_t bal = __ballot_sync(0xffffffffu, perfect);
      if (lane == 0) s_warp[warp] = __popc(bal);
      __syncthreads();
      int rank = before + __popc(bal & ((1u << lane) - 1u));
      for (int w = 0; w < nt >> 5; ++w) {
        if (w < warp) rank += s_warp[w];
        before += s_warp[w];
      }
      if (i < g.n) {
        const bool chosen = perfect && rank < k;
        pruned[g.lo + i] = chosen ? 0 : 1;
        if (chosen) out[rank] = g.lo + i;
      }
      __syncthreads();
    }
    if (tid == 0) final_out[blockIdx.x] = 1;
    return;
  }
  const bool all_verified = nver == g.n;
  for (int j = (all_verified ? nver : 0) + tid; j < k; j += nt) out[j] = -1;
  sorted(g.n, smem_keys, scratch + 2 * static_cast<int64_t>(g.lo),
         [&](int i) {                             // (an unverified one: behind every score's key, a NaN's too, still distinct)
           return verified[g.lo + i] ? make_key(scores[g.lo + i], static_cast<uint32_t>(i)) : kUnverified | static_cast<uint32_t>(i);
         },
         [&](int j, uint64_t key) {
           const int cand = g.lo + static_cast<int>(key & 0x7fffffffu);
           pruned[cand] = j < nver && nver > k && j >= k ? 1 : 0;
           if (all_verified && j < k) out[j] = cand;
         });
  if (tid == 0) final_out[blockIdx.x] = all_verified ? 1 : 0;
}
__global__ void __launch_bounds__(kMaxThreads)
early_prune_kernel(const float* __restrict__ scores, const uint8_t* __restrict__ verified,
                   const int32_t* __restrict__ seg_offsets, int n_total, int k, uint8_t* __restrict__ pruned,
                   int32_t* __restrict__ selected, uint8_t* __restrict__ final_out, uint64_t* __restrict__ scratch,
                   int32_t* __restrict__ status) {
  ss::grid_dependency_enter();
  __shared__ uint64_t smem_keys[kSmemKeys];
  __shared__ int s_nver, s_nperfect;
  if (threadIdx.x == 0) { s_nver = 0; s_nperfect = 0; }
  const Segment g = open_segment(blockIdx.x, gridDim.x, seg_offsets, n_total, pruned, status);
  early_prune_segment(scores, verified, g, k, pruned, selected, final_out, scratch, smem_keys, s_nver, s_nperfect);
  if (g.gaps) clear_uncovered(seg_offsets, gridDim.x, n_total, pruned, smem_keys);
}

}  // namespace topk
}  // namespace ss

extern "C" int32_t ss_early_prune(const float* scores, const uint8_t* verified, const int32_t* seg_offsets,
                                  int32_t n_segments, int32_t n_total, int32_t k, uint8_t* pruned_out,
                                  int32_t* selected_out, uint8_t* final_out, void* workspace, size_t workspace_bytes,
                                  void* stream) {
  using namespace ss;
  if (n_segments < 0 || n_total < 0 || k < 1) return SS_ERR_INVALID_ARG;
  cudaStream_t st = as_stream(stream);
  if (n_segments == 0) {
    if (n_total > 0 && pruned_out && cudaMemsetAsync(pruned_out, 0, static_cast<size_t>(n_total), st) != cudaSuccess) {
      (void)cudaGetLastError();
      return SS_ERR_CUDA;
    }
    return SS_OK;
  }
  if (!seg_offsets || !selected_out || !final_out || !workspace) return SS_ERR_INVALID_ARG;
  if (n_total > 0 && (!scores || !verified || !pruned_out)) return SS_ERR_INVALID_ARG;
  if (reinterpret_cast<uintptr_t>(workspace) % kAlign) return SS_ERR_INVALID_ARG;
  size_t need = 0;
  ss_topk_workspace_bytes(n_total, &need);
  if (workspace_bytes < need) return SS_ERR_WORKSPACE_TOO_SMALL;
  SS_LAUNCH(topk::early_prune_kernel, n_segments, topk::block_threads(n_total, n_segments), 0, st, scores, verified, seg_offsets, n_total, k,
            pruned_out, selected_out, final_out, reinterpret_cast<uint64_t*>(static_cast<char*>(workspace) + kAlign),
            static_cast<int32_t*>(workspace));
  return SS_OK;
}

extern "C" int32_t ss_topk_workspace_bytes(int32_t n_total, size_t* out_bytes) {
  if (n_total < 0 || !out_bytes) return SS_ERR_INVALID_ARG;
  // the status word (first bytes, see ss_last_device_status), then two 64-bit sort keys per candidate
  *out_bytes = ss::kAlign + ss::align_up(static_cast<size_t>(2) * (n_total > 0 ? n_total : 1) * sizeof(uint64_t));
  return SS_OK;
}

extern "C" int32_t ss_topk_prune(const float* scores, const int32_t* seg_offsets, int32_t n_segments,
                                 int32_t n_total, int32_t k, int32_t* survivors_out, uint8_t* keep_out,
                                 void* workspace, size_t workspace_bytes, void* stream) {
  using namespace ss;
  if (n_segments < 0 || n_total < 0 || k < 1) return SS_ERR_INVALID_ARG;
  if (n_segments == 0) {
    if (n_total > 0 && keep_out &&
        cudaMemsetAsync(keep_out, 0, static_cast<size_t>(n_total), as_stream(stream)) != cudaSuccess) {
      (void)cudaGetLastError();
      return SS_ERR_CUDA;
    }
    return SS_OK;
  }
  if (!seg_offsets || !survivors_out || !workspace) return SS_ERR_INVALID_ARG;
  if (n_total > 0 && (!scores || !keep_out)) return SS_ERR_INVALID_ARG;
  if (reinterpret_cast<uintptr_t>(workspace) % kAlign) return SS_ERR_INVALID_ARG;
  size_t need = 0;
  ss_topk_workspace_bytes(n_total, &need);
  if (workspace_bytes < need) return SS_ERR_WORKSPACE_TOO_SMALL;
  cudaStream_t st = as_stream(stream);
  SS_LAUNCH(topk::topk_kernel, n_segments, topk::block_threads(n_total, n_segments), 0, st, scores, seg_offsets, n_total, k, survivors_out, keep_out,
            reinterpret_cast<uint64_t*>(static_cast<char*>(workspace) + kAlign), static_cast<int32_t*>(workspace));
  return SS_OK;
}
