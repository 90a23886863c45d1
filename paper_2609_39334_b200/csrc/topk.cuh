// Selection by score: what a block does with its segment (ss_topk_prune, ss_early_prune and the front of a device step).
#pragma once
#include "common.cuh"

namespace ss {
namespace topk {

constexpr int kMaxThreads = 1024;
constexpr int kSmemKeys = 4096;     // 32 KB of shared memory
constexpr uint64_t kUnverified = 0xffffffff80000000ull;   // | index: a NaN's key has the same high word, bit 31 clear

__device__ __forceinline__ uint64_t make_key(float f, uint32_t local_idx) {
  uint32_t ordered;                           // ascending in the score
  if (f != f) {
    ordered = 0u;                             // NaN below every number (below -inf, whose code is 0x007fffff)
  } else {
    f = f + 0.0f;                             // -0.0 -> +0.0
    const uint32_t u = __float_as_uint(f);
    ordered = (u & 0x80000000u) ? ~u : (u | 0x80000000u);
  }
  return (static_cast<uint64_t>(~ordered) << 32) | local_idx;
}

__device__ __forceinline__ void bitonic_sort(uint64_t* keys, int n_pad) {
  for (int size = 2; size <= n_pad; size <<= 1) {
    for (int stride = size >> 1; stride > 0; stride >>= 1) {
      for (int t = threadIdx.x; t < (n_pad >> 1); t += blockDim.x) {
        const int lo = ((t / stride) * (stride << 1)) + (t % stride);
        const int hi = lo + stride;
        const bool up = ((lo & size) == 0);
        const uint64_t a = keys[lo], b = keys[hi];
        if ((a > b) == up) { keys[lo] = b; keys[hi] = a; }
      }
      __syncthreads();
    }
  }
}

// One key per thread (n_pad <= blockDim.x, a power of two): returns the key of rank threadIdx.x.  Threads past n_pad bring
// padding (~0) and keep it.
__device__ __forceinline__ uint64_t sort_registers(uint64_t k, int n_pad, uint64_t* s_key) {
  const int tid = threadIdx.x;
  for (int size = 2; size <= n_pad; size <<= 1) {
    for (int stride = size >> 1; stride > 0; stride >>= 1) {
      uint64_t other;
      if (stride >= 32) {
        s_key[tid] = k;
        __syncthreads();
        other = s_key[tid ^ stride];
        __syncthreads();
      } else {
        other = __shfl_xor_sync(0xffffffffu, k, stride);
      }
      const bool keep_low = ((tid & stride) == 0) == ((tid & size) == 0);
      if ((k > other) == keep_low) k = other;
    }
  }
  return k;
}

// A block's segment.  One that does not lie inside [0, n_total] is reported and treated as empty: its offsets index the mask
// and the scratch region, so following them would write out of bounds.  The first segment's block looks at all segments, writes the status word
// and clears `mask` where NO valid segment lies, so that it never writes what another block does: in front of the first and
// behind the last one here, or, with a bad one among them (`gaps`), by clear_uncovered when its own segment is done - not
// before: the compiler then makes the sort slower for everybody (512 segments of 1024: 31.9 us instead of 25.0).
struct Segment {
  int lo, n;
  bool gaps;
};
__device__ __forceinline__ bool valid_segment(int lo, int hi, int n_total) { return lo >= 0 && hi >= lo && hi <= n_total; }
static __device__ __noinline__ void clear_uncovered(const int32_t* __restrict__ seg_offsets, int n_segments, int n_total, uint8_t* mask,
                                             uint64_t* smem_keys) {
  constexpr int kWindow = kSmemKeys * 64;                     // candidates a pass, a bit each
  uint32_t* covered = reinterpret_cast<uint32_t*>(smem_keys);
  const int tid = threadIdx.x, nt = blockDim.x;
  __syncthreads();
  for (int base = 0; base < n_total; base = base > n_total - kWindow ? n_total : base + kWindow) {
    const int end = n_total - base < kWindow ? n_total : base + kWindow;
    for (int i = tid; i < kWindow / 32; i += nt) covered[i] = 0;
    __syncthreads();
    for (int x = tid; x < n_segments; x += nt) {
      if (!valid_segment(seg_offsets[x], seg_offsets[x + 1], n_total)) continue;
      const int l = max(seg_offsets[x], base) - base, h = min(seg_offsets[x + 1], end) - base;
      for (int w = l >> 5; l < h && w <= (h - 1) >> 5; ++w) {
        const uint32_t from = 0xffffffffu << (w == l >> 5 ? l & 31 : 0), to = 0xffffffffu >> (w == (h - 1) >> 5 ? 31 - ((h - 1) & 31) : 0);
        atomicOr(&covered[w], from & to);
      }
    }
    __syncthreads();
    for (int i = tid; i < end - base; i += nt)
      if (!((covered[i >> 5] >> (i & 31)) & 1u)) mask[base + i] = 0;
    __syncthreads();
  }
}
__device__ __forceinline__ Segment open_segment(int s, int n_segments, const int32_t* __restrict__ seg_offsets, int n_total,
                                                uint8_t* mask, int32_t* status) {
  const int nt = blockDim.x;
  const int lo = seg_offsets[s], hi = seg_offsets[s + 1];
  bool any = false;
  if (s == 0) {
    const int tail = seg_offsets[n_segments];                 // (loaded with the others, not behind the barrier)
    for (int x = threadIdx.x; x < n_segments; x += nt) any = any || !valid_segment(seg_offsets[x], seg_offsets[x + 1], n_total);
    any = __syncthreads_or(any) != 0;
    if (threadIdx.x == 0) *status = any ? SS_ERR_BAD_INPUT : SS_OK;
    if (!any) {
      for (int i = threadIdx.x; i < lo; i += nt) mask[i] = 0;
      for (int i = tail + static_cast<int>(threadIdx.x); i < n_total; i += nt) mask[i] = 0;
    }
  }
  return Segment{lo, valid_segment(lo, hi, n_total) ? hi - lo : 0, any};
}

// Calls rank(j, key) for the key of every rank j < n, n keys from make(i).  `scratch`: where neither the registers nor
// shared memory take the segment.
template <typename Make, typename Rank>
__device__ __forceinline__ void sorted(int n, uint64_t* smem_keys, uint64_t* scratch, Make make, Rank rank) {
  int n_pad = 1;
  while (n_pad < n) n_pad <<= 1;
  const int tid = threadIdx.x, nt = blockDim.x;
  if (n_pad <= nt) {
    const uint64_t k = sort_registers(tid < n ? make(tid) : ~0ull, n_pad, smem_keys);
    if (tid < n) rank(tid, k);
    return;
  }
  uint64_t* keys = n_pad <= kSmemKeys ? smem_keys : scratch;
  for (int i = tid; i < n_pad; i += nt) keys[i] = i < n ? make(i) : ~0ull;
  __syncthreads();
  bitonic_sort(keys, n_pad);
  for (int j = tid; j < n; j += nt) rank(j, keys[j]);
}

// A block: segment s of n_segments, its k best and its part of the mask.
__device__ __forceinline__ void select_segment(int s, int n_segments, const float* __restrict__ scores, const int32_t* __restrict__ seg_offsets,
                                               int n_total, int k, int32_t* __restrict__ survivors, uint8_t* __restrict__ keep,
                                               uint64_t* __restrict__ scratch, int32_t* __restrict__ status, uint64_t* smem_keys) {
  const Segment g = open_segment(s, n_segments, seg_offsets, n_total, keep, status);
  int32_t* out = survivors + static_cast<int64_t>(s) * k;
  for (int j = g.n + threadIdx.x; j < k; j += blockDim.x) out[j] = -1;
  // (a segment's scratch region starts at 2 lo: pow2ceil(n) < 2n keeps the regions of different segments apart)
  if (g.n > 0)
    sorted(g.n, smem_keys, scratch + 2 * static_cast<int64_t>(g.lo),
           [&](int i) { return make_key(scores[g.lo + i], static_cast<uint32_t>(i)); },
           [&](int j, uint64_t key) {
             const int cand = g.lo + static_cast<int>(key & 0xffffffffu);
             keep[cand] = j < k ? 1 : 0;
             if (j < k) out[j] = cand;
           });
  if (g.gaps) clear_uncovered(seg_offsets, n_segments, n_total, keep, smem_keys);
}

// Threads per block: one per candidate of a segment of average size, but more where there are so many candidates, since any one
// segment may be far above the average: one of 4096 among 1000 of 16 takes 236 us with 64 threads and 76 with 256.  Few
// candidates get 128: a decode step of 16 segments of 64 takes 1 us more with 256 (107.0 us, 106.1 with 64 or 128), whose blocks
// are in the way of the kernels around them.  512 segments of 16: 2.6 us with 64, 3.3 with 256.
inline int block_threads(int n_total, int n_segments) {
  const int least = n_total <= 2048 ? 128 : 256;
  int t = 64;
  while (t < least && t < n_total) t <<= 1;
  while (t < kMaxThreads && static_cast<int64_t>(t) * n_segments < n_total) t <<= 1;
  return t;
}

}  // namespace topk
}  // namespace ss
