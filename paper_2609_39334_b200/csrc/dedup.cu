// ss_dedup_paths: computation deduplication of candidate paths (paper, Section "Computation Deduplication").
//
// Pipeline (all on the caller's stream, no host synchronisation):
//   1. hash      one warp per path: 64-bit hash of (ctx_key, length, token ids); lanes stride over the tokens,
//                each token is mixed with its position, lane sums are combined with shuffles
//   2. table     open addressing, one entry per distinct hash: the smallest path index with it
//   3. match     one warp per path: compares itself with the path of its entry - 64-bit hash, ctx_key, length AND token ids
//                (by the whole warp) -> canon.  If they differ the hash collided, and the warp looks through all earlier
//                paths with an equal hash.
//   4. compact   exclusive scan of (canon[i] == i) in index order -> ranks; unique list, multiplicities (counts:
//                order-independent), path_to_unique, slot remap
// Hash collisions only cost time: equality is always decided on the token ids themselves.
//
// Up to kClusterMax paths this is one launch of a cluster.  Up to kSmallMax paths it takes two launches and no cleared memory: every block of the second builds the whole table in
// its own shared memory (a microsecond; cheaper than a launch that builds it once), matches its 32 paths, and the block
// that arrives last compacts.  Above, the first launch inserts into a table in the workspace, the second matches, and the
// third compacts with a block per 1024 paths.  Latency-bound: a few MB of ids, a handful of dependent trips to L2.
// Measured, the call: 1024 paths 35 -> 14 us (a bitonic sort of the hashes and binary searches by one block before),
// 8192 paths 78 -> 28 us (a sort by counting, a compaction by one block).
#include "step.cuh"
#include "topk.cuh"

namespace ss {
namespace dedup {

constexpr int kThreads = 1024;                      // match kernels: a warp per path
constexpr int kWarps = kThreads / 32;
constexpr int kSmallMax = 4096;
constexpr int kHashWarps = 8;                       // per block of the hash kernels
constexpr int kChunk = 1024;                        // paths per block of the compaction

__device__ __forceinline__ uint64_t mix64(uint64_t x) {   // splitmix64 finaliser
  x ^= x >> 30; x *= 0xbf58476d1ce4e5b9ull;
  x ^= x >> 27; x *= 0x94d049bb133111ebull;
  x ^= x >> 31;
  return x;
}

// Ids of a path that a lane has on their way.  Up to kSmallMax paths wait for memory: with eight, paths of 300 tokens are two trips,
// not ten (the step of 1024 paths 78.4 us, 83.5 with four; 4096 paths of up to 2000 tokens 29 us, 45 with one, 34 with a test for
// each of eight).  More paths are bound by instructions and registers: 100000 of up to 300 tokens 96 us with four, 113 with eight.
// Whole rounds go without a test for each id, and a warp leaves a round where nothing is left: 100000 of up to 8 tokens 57 us, 85
// with a test for each of eight, 59 with one id at a time.
constexpr int kAheadSmall = 8, kAheadLarge = 4;
constexpr uint64_t kId = 0x9e3779b97f4a7c15ull, kAt = 0xd1b54a32d192ed03ull;
// Whole warp: 64-bit hash of path `path` (returned to every lane).
template <int kAhead>
__device__ __forceinline__ uint64_t hash_path(const int32_t* __restrict__ tok_ids, const int64_t* __restrict__ tok_offsets,
                                              const int64_t* __restrict__ ctx_key, int path, uint32_t weak, int lane) {
  const int64_t lo = tok_offsets[path], hi = tok_offsets[path + 1];
  uint64_t acc = 0, at = static_cast<uint64_t>(lane + 1) * kAt;   // (position + 1) * kAt
  const int32_t* p = tok_ids + lo + lane;
  int64_t left = hi - lo;
  for (; left >= 32 * kAhead; left -= 32 * kAhead, p += 32 * kAhead, at += 32 * kAhead * kAt) {
    uint32_t t[kAhead];
#pragma unroll
    for (int u = 0; u < kAhead; ++u) t[u] = static_cast<uint32_t>(p[32 * u]);
#pragma unroll
    for (int u = 0; u < kAhead; ++u) acc += mix64(t[u] * kId + at + 32 * u * kAt);
  }
  const int rest = static_cast<int>(left);
  uint32_t t[kAhead];
#pragma unroll
  for (int u = 0; u < kAhead; ++u) {                        // (the warp leaves where nothing is left: most paths have a few tokens)
    if (kAhead == kAheadLarge && 32 * u >= rest) break;
    t[u] = lane + 32 * u < rest ? static_cast<uint32_t>(p[32 * u]) : 0u;
  }
#pragma unroll
  for (int u = 0; u < kAhead; ++u) {
    if (32 * u >= rest) break;
    const uint64_t m = mix64(t[u] * kId + at + 32 * u * kAt);
    if (lane + 32 * u < rest) acc += m;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  uint64_t h = mix64(acc ^ mix64(static_cast<uint64_t>(hi - lo) + 0x632be59bd9b4e019ull));
  if (ctx_key) h = mix64(h ^ mix64(static_cast<uint64_t>(ctx_key[path]) + 0x2545f4914f6cdd1dull));
  if (weak) h &= 0xffull;                       // SS_FLAG_WEAK_HASH: force collisions
  return h;
}

// Entry of the table in the workspace: tag << 32 | smallest path index; all ones when empty.
constexpr unsigned long long kEmpty = ~0ull;
__device__ __forceinline__ uint32_t tag_of(uint64_t h) { return static_cast<uint32_t>(h >> 32) ^ static_cast<uint32_t>(h); }

// Hash of every path.  `table` (mask + 1 entries, all ones): inserts; `chunk_count`, `multiplicity`: cleared for the kernels
// that follow; `arrived`: the counter of small_match_kernel.
template <int kAhead>
__global__ void hash_kernel(const int32_t* __restrict__ tok_ids, const int64_t* __restrict__ tok_offsets,
                            const int64_t* __restrict__ ctx_key, int n, uint32_t weak, uint64_t* __restrict__ hash64,
                            unsigned long long* table, uint32_t mask, int* __restrict__ chunk_count,
                            int32_t* __restrict__ multiplicity, unsigned int* __restrict__ arrived) {
  ss::grid_dependency_enter();
  const int lane = threadIdx.x & 31;
  const int64_t gtid = static_cast<int64_t>(blockIdx.x) * (kHashWarps * 32) + threadIdx.x;
  if (gtid == 0 && arrived) *arrived = 0;
  if (table && gtid < n) {
    multiplicity[gtid] = 0;
    if (gtid % kChunk == 0) chunk_count[gtid / kChunk] = 0;
  }
  if ((gtid >> 5) >= n) return;
  const int path = static_cast<int>(gtid >> 5);
  const uint64_t h = hash_path<kAhead>(tok_ids, tok_offsets, ctx_key, path, weak, lane);
  if (lane != 0) return;
  hash64[path] = h;
  if (!table) return;
  const unsigned long long mine = (static_cast<unsigned long long>(tag_of(h)) << 32) | static_cast<uint32_t>(path);
  for (uint32_t s = static_cast<uint32_t>(h) & mask;; s = (s + 1) & mask) {
    // (the entry is looked at first: of many equal paths most then find a smaller one there.  With the counts below: 1M equal paths
    //  3.0 -> 0.5 ms; different ones 0.54 either way)
    unsigned long long cur = __ldcg(&table[s]);
    if (cur == kEmpty) cur = atomicCAS(&table[s], kEmpty, mine);
    if (cur == kEmpty) return;
    if ((cur >> 32) == (mine >> 32)) {                       // (an entry keeps its tag: the minimum is over the index)
      if (cur > mine) atomicMin(&table[s], mine);
      return;
    }
  }
}

// The selection of a step, which needs nothing from the deduplication nor it from the selection: blocks of the first launch.
struct Selection {
  const float* scores;
  const int32_t* seg_offsets;
  int n_segments, k;
  int32_t* survivors;
  uint8_t* keep;
  uint64_t* scratch;
  int32_t* status;
};
__device__ __forceinline__ void selection_block(const Selection& T, int s, int n) {
  __shared__ uint64_t smem_keys[topk::kSmemKeys];
  topk::select_segment(s, T.n_segments, T.scores, T.seg_offsets, n, T.k, T.survivors, T.keep, T.scratch, T.status, smem_keys);
}
// Hash of every path, as above without a table, and the selection's blocks behind those of the hash.
__global__ void __launch_bounds__(kHashWarps * 32)
hash_select_kernel(const int32_t* __restrict__ tok_ids, const int64_t* __restrict__ tok_offsets,
                   const int64_t* __restrict__ ctx_key, int n, uint32_t weak, uint64_t* __restrict__ hash64,
                   unsigned int* __restrict__ arrived, int hash_blocks, const __grid_constant__ Selection T) {
  ss::grid_dependency_enter();
  if (static_cast<int>(blockIdx.x) >= hash_blocks) {
    selection_block(T, blockIdx.x - hash_blocks, n);
    return;
  }
  const int lane = threadIdx.x & 31, path = blockIdx.x * kHashWarps + (threadIdx.x >> 5);
  if (blockIdx.x == 0 && threadIdx.x == 0) *arrived = 0;
  if (path >= n) return;
  const uint64_t h = hash_path<kAheadSmall>(tok_ids, tok_offsets, ctx_key, path, weak, lane);
  if (lane == 0) hash64[path] = h;
}

// Whole warp: paths i and j have the same context, length and ids.
template <int kAhead>
__device__ __forceinline__ bool same_path(const int32_t* __restrict__ tok_ids, const int64_t* __restrict__ tok_offsets,
                                          const int64_t* __restrict__ ctx_key, int i, int j, int lane) {
  const int64_t a0 = tok_offsets[i], b0 = tok_offsets[j], len = tok_offsets[i + 1] - a0;
  if (tok_offsets[j + 1] - b0 != len || (ctx_key && ctx_key[i] != ctx_key[j])) return false;
  const int32_t *a = tok_ids + a0 + lane, *b = tok_ids + b0 + lane;
  int64_t left = len;
  for (; left >= 32 * kAhead; left -= 32 * kAhead, a += 32 * kAhead, b += 32 * kAhead) {
    int32_t x[kAhead], y[kAhead];
#pragma unroll
    for (int u = 0; u < kAhead; ++u) {
      x[u] = a[32 * u];
      y[u] = b[32 * u];
    }
    int32_t diff = 0;
#pragma unroll
    for (int u = 0; u < kAhead; ++u) diff |= x[u] ^ y[u];
    if (__any_sync(0xffffffffu, diff != 0)) return false;
  }
  const int rest = static_cast<int>(left);
  int32_t x[kAhead], y[kAhead];
#pragma unroll
  for (int u = 0; u < kAhead; ++u) {
    x[u] = y[u] = 0;
    if (lane + 32 * u < rest) {
      x[u] = a[32 * u];
      y[u] = b[32 * u];
    }
  }
  int32_t diff = 0;
#pragma unroll
  for (int u = 0; u < kAhead; ++u) diff |= x[u] ^ y[u];
  return !__any_sync(0xffffffffu, diff != 0);
}

// Whole warp: canonical representative of path i, given the smallest path j <= i in its table entry.
template <int kAhead>
__device__ __forceinline__ int canon_of(const int32_t* __restrict__ tok_ids, const int64_t* __restrict__ tok_offsets,
                                        const int64_t* __restrict__ ctx_key, const uint64_t* hash64, uint64_t h, int i, int j,
                                        int lane) {
  if (j == i || (hash64[j] == h && same_path<kAhead>(tok_ids, tok_offsets, ctx_key, i, j, lane))) return j;
  for (int b = 0; b < i; b += 32) {                           // a collision
    const int t = b + lane;
    uint32_t m = __ballot_sync(0xffffffffu, t < i && t != j && hash64[t < i ? t : 0] == h);
    while (m) {
      const int c = b + __ffs(m) - 1;
      m &= m - 1;
      if (same_path<kAhead>(tok_ids, tok_offsets, ctx_key, i, c, lane)) return c;
    }
  }
  return i;
}

// True in every thread of the block that arrives last; its reads come after all other blocks' writes.
__device__ __forceinline__ bool last_block_arrives(unsigned int* counter) {
  __shared__ bool s_last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) s_last = atomicAdd(counter, 1u) == gridDim.x - 1;
  __syncthreads();
  if (s_last) __threadfence();
  return s_last;
}

// ---- up to kSmallMax paths ---------------------------------------------------------------------------------------
inline int small_table_size(int n) {
  int t = 64;
  while (t < 2 * n) t <<= 1;
  return t;
}
inline size_t small_match_smem(int n) { return static_cast<size_t>(n) * 8 + static_cast<size_t>(small_table_size(n)) * 4; }

// Table of all paths in the block's shared memory (s_hash[n], s_tab[mask + 1]), then the canonical representatives of the
// paths blockIdx.x * kWarps + warp, every `step`-th from there.
__device__ __forceinline__ void small_match(const int32_t* __restrict__ tok_ids, const int64_t* __restrict__ tok_offsets,
                                            const int64_t* __restrict__ ctx_key, int n, const uint64_t* hash64,
                                            int32_t* canon_out, uint64_t* s_hash, int* s_tab, uint32_t mask, int step) {
  const int tid = threadIdx.x, lane = tid & 31;
  for (int i = tid; i < n; i += kThreads) s_hash[i] = __ldcg(hash64 + i);
  for (int t = tid; t <= static_cast<int>(mask); t += kThreads) s_tab[t] = -1;
  __syncthreads();
  for (int i = tid; i < n; i += kThreads) {
    const uint64_t h = s_hash[i];
    for (uint32_t s = static_cast<uint32_t>(h) & mask;; s = (s + 1) & mask) {
      const int cur = atomicCAS(&s_tab[s], -1, i);
      if (cur < 0) break;
      if (s_hash[cur] == h) {
        atomicMin(&s_tab[s], i);
        break;
      }
    }
  }
  __syncthreads();
  for (int i = blockIdx.x * kWarps + (tid >> 5); i < n; i += step) {
    const uint64_t h = s_hash[i];
    uint32_t s = static_cast<uint32_t>(h) & mask;
    while (s_hash[s_tab[s]] != h) s = (s + 1) & mask;
    const int c = canon_of<kAheadSmall>(tok_ids, tok_offsets, ctx_key, s_hash, h, i, s_tab[s], lane);
    if (lane == 0) canon_out[i] = c;
  }
}

// The descriptor rows of the unique paths (see gather_unique_kernel), made with the compaction where a whole step is one call.
struct Gather {
  const int32_t *path_leaf_node, *path_q_len;
  const int64_t* q_offsets;
  int32_t *u_leaf, *u_q_len;                                  // null: no gather
  int64_t *u_q_offsets, *u_q_src;
};
constexpr int kOwn = kSmallMax / kThreads;                    // paths of a thread: tid, tid + kThreads, ...
// A path's own descriptor row, loaded before it is known whether it is wanted (all blocks do, the last one needs them).
struct GatherRows {
  int leaf[kOwn], len[kOwn];
  int64_t src[kOwn];
};
template <bool GATHER>
__device__ __forceinline__ void load_rows(GatherRows& R, const Gather& G, int n) {
  if (!GATHER) return;
#pragma unroll
  for (int e = 0; e < kOwn; ++e) {
    const int i = threadIdx.x + e * kThreads;
    R.leaf[e] = i < n ? G.path_leaf_node[i] : -1;
    R.len[e] = i < n ? G.path_q_len[i] : 0;
    R.src[e] = i < n ? G.q_offsets[i] : 0;
  }
}

// One block, all of canon_out written: ranks, unique list, multiplicities, remap (and the gather).  s_mem: 8 n bytes.
template <bool GATHER>
__device__ __forceinline__ void small_compact(int n, const int32_t* __restrict__ slot_in, const int32_t* canon_out,
                                              int32_t* path_to_unique, int32_t* unique_paths, int32_t* multiplicity,
                                              int32_t* slot_out, int32_t* num_unique, uint8_t* s_mem, const Gather& G,
                                              const GatherRows& R) {
  __shared__ int s_before[kSmallMax / 32];                    // unique paths in front of each group of 32
  __shared__ long long s_rows[GATHER ? kSmallMax / 32 : 1], s_all_rows;   // and their query rows
  __shared__ int s_total;
  const int tid = threadIdx.x, lane = tid & 31, groups = (n + 31) >> 5;
  int* s_rank = reinterpret_cast<int*>(s_mem);
  int* s_mult = s_rank + n;
  int canon[kOwn];
  long long rows[kOwn];                                       // of the unique paths up to this one in its group
#pragma unroll
  for (int e = 0; e < kOwn; ++e) {
    const int i = tid + e * kThreads;
    canon[e] = i < n ? __ldcg(canon_out + i) : -1;
  }
#pragma unroll
  for (int e = 0; e < kOwn; ++e) {
    const int i = tid + e * kThreads;
    if (i - lane >= n) break;
    const uint32_t u = __ballot_sync(0xffffffffu, canon[e] == i);
    if (i < n) {
      s_rank[i] = __popc(u & ((1u << lane) - 1u));
      s_mult[i] = 0;
    }
    if (lane == 0) s_before[i >> 5] = __popc(u);
    if (GATHER) {
      rows[e] = canon[e] == i ? R.len[e] : 0;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const long long y = __shfl_up_sync(0xffffffffu, rows[e], o);
        if (lane >= o) rows[e] += y;
      }
      if (lane == 31) s_rows[i >> 5] = rows[e];
    }
  }
  __syncthreads();
  if (tid < 32) {                                             // 4 groups a lane
    int v[4], sum = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      v[k] = 4 * lane + k < groups ? s_before[4 * lane + k] : 0;
      sum += v[k];
    }
    int incl = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += y;
    }
    int run = incl - sum;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      if (4 * lane + k < groups) s_before[4 * lane + k] = run;
      run += v[k];
    }
    if (lane == 31) s_total = incl;
  } else if (GATHER && tid < 64) {
    long long v[4], sum = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      v[k] = 4 * lane + k < groups ? s_rows[4 * lane + k] : 0;
      sum += v[k];
    }
    long long incl = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const long long y = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += y;
    }
    long long run = incl - sum;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      if (4 * lane + k < groups) s_rows[4 * lane + k] = run;
      run += v[k];
    }
    if (lane == 31) s_all_rows = incl;
  }
  __syncthreads();
  const int total = s_total;
#pragma unroll
  for (int e = 0; e < kOwn; ++e) {
    const int i = tid + e * kThreads;
    if (i >= n) break;
    const int c = canon[e], r = s_before[c >> 5] + s_rank[c];
    path_to_unique[i] = r;
    if (c == i) unique_paths[r] = i;
    atomicAdd(&s_mult[r], 1);
    if (slot_out) slot_out[i] = slot_in[c];
    if (GATHER) {
      if (c == i) {
        G.u_leaf[r] = R.leaf[e];
        G.u_q_len[r] = R.len[e];
        G.u_q_src[r] = R.src[e];
        G.u_q_offsets[r + 1] = s_rows[i >> 5] + rows[e];
      }
      if (i >= total) {                                       // inert entries
        G.u_leaf[i] = -1;
        G.u_q_len[i] = 0;
        G.u_q_src[i] = 0;
        G.u_q_offsets[i + 1] = s_all_rows;
      }
    }
  }
  if (GATHER && tid == 0) G.u_q_offsets[0] = 0;
  __syncthreads();
  for (int i = tid; i < total; i += kThreads) multiplicity[i] = s_mult[i];
  for (int i = total + tid; i < n; i += kThreads) multiplicity[i] = 0;
  if (tid == 0) *num_unique = total;
}

template <bool GATHER>
__global__ void __launch_bounds__(kThreads)
small_match_kernel(const int32_t* __restrict__ tok_ids, const int64_t* __restrict__ tok_offsets,
                   const int64_t* __restrict__ ctx_key, int n, const uint64_t* __restrict__ hash64, uint32_t mask,
                   const int32_t* __restrict__ slot_in, int32_t* canon_out, int32_t* path_to_unique, int32_t* unique_paths,
                   int32_t* multiplicity, int32_t* slot_out, int32_t* num_unique, unsigned int* arrived,
                   const __grid_constant__ Gather G) {
  ss::grid_dependency_enter();
  extern __shared__ __align__(16) uint8_t s_mem[];
  uint64_t* s_hash = reinterpret_cast<uint64_t*>(s_mem);
  GatherRows R;
  load_rows<GATHER>(R, G, n);
  small_match(tok_ids, tok_offsets, ctx_key, n, hash64, canon_out, s_hash, reinterpret_cast<int*>(s_hash + n), mask, n);
  if (!last_block_arrives(arrived)) return;
  // compaction by the last block; the hashes' shared memory holds ranks and multiplicities
  small_compact<GATHER>(n, slot_in, canon_out, path_to_unique, unique_paths, multiplicity, slot_out, num_unique, s_mem, G, R);
}

// ---- up to kClusterMax paths: one launch of one cluster, whose barrier separates hash, match and compaction -------------
// Kernel time in a graph, cluster against two launches: 8 paths of 64 tokens 5.2 / 5.7 us, 72 of one token 6.1 / 6.2, 128 of
// 300 tokens 9.8 / 8.4, 1024 of 300 20.9 / 11.8; the second launch costs the host 2.3 us.
constexpr int kClusterMax = 96;
constexpr int kClusterBlocks = 8;
__device__ __forceinline__ void cluster_barrier() {
  asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}
// STEP: with the gather, and the selection by the clusters behind the first.
template <bool STEP>
__global__ void __cluster_dims__(kClusterBlocks, 1, 1) __launch_bounds__(kThreads)
cluster_dedup_kernel(const int32_t* __restrict__ tok_ids, const int64_t* __restrict__ tok_offsets,
                     const int64_t* __restrict__ ctx_key, int n, uint32_t weak, uint64_t* hash64, uint32_t mask,
                     const int32_t* __restrict__ slot_in, int32_t* canon_out, int32_t* path_to_unique, int32_t* unique_paths,
                     int32_t* multiplicity, int32_t* slot_out, int32_t* num_unique, const __grid_constant__ Gather G,
                     const __grid_constant__ Selection T) {
  ss::grid_dependency_enter();
  if (STEP && blockIdx.x >= kClusterBlocks) {
    if (static_cast<int>(blockIdx.x) - kClusterBlocks < T.n_segments) selection_block(T, blockIdx.x - kClusterBlocks, n);
    return;
  }
  __shared__ __align__(16) uint64_t s_hash[kClusterMax];
  __shared__ int s_tab[4 * kClusterMax];                        // (small_table_size: below 4 n, at least 64)
  const int lane = threadIdx.x & 31;
  GatherRows R;
  load_rows<STEP>(R, G, n);
  for (int i = blockIdx.x * kWarps + (threadIdx.x >> 5); i < n; i += kClusterBlocks * kWarps) {
    const uint64_t h = hash_path<kAheadSmall>(tok_ids, tok_offsets, ctx_key, i, weak, lane);
    if (lane == 0) hash64[i] = h;
  }
  cluster_barrier();
  small_match(tok_ids, tok_offsets, ctx_key, n, hash64, canon_out, s_hash, s_tab, mask, kClusterBlocks * kWarps);
  cluster_barrier();
  if (blockIdx.x == 0)
    small_compact<STEP>(n, slot_in, canon_out, path_to_unique, unique_paths, multiplicity, slot_out, num_unique,
                        reinterpret_cast<uint8_t*>(s_hash), G, R);
}

// ---- more paths -----------------------------------------------------------------------------------------------------
// unique[w]: bit b set if path 32 w + b is its own representative; chunk_count[c]: how many of chunk c are.
__global__ void __launch_bounds__(kThreads)
match_kernel(const int32_t* __restrict__ tok_ids, const int64_t* __restrict__ tok_offsets, const int64_t* __restrict__ ctx_key,
             int n, const uint64_t* __restrict__ hash64, const unsigned long long* __restrict__ table, uint32_t mask,
             int32_t* __restrict__ canon_out, uint32_t* __restrict__ unique, int* chunk_count) {
  ss::grid_dependency_enter();
  __shared__ int s_own[kWarps];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, i = blockIdx.x * kWarps + warp;
  int own = 0;
  if (i < n) {
    const uint64_t h = hash64[i];
    const uint32_t tag = tag_of(h);
    uint32_t s = static_cast<uint32_t>(h) & mask;
    unsigned long long e = table[s];
    while (static_cast<uint32_t>(e >> 32) != tag) {
      s = (s + 1) & mask;
      e = table[s];
    }
    const int c = canon_of<kAheadLarge>(tok_ids, tok_offsets, ctx_key, hash64, h, i, static_cast<int>(static_cast<uint32_t>(e)), lane);
    if (lane == 0) canon_out[i] = c;
    own = c == i ? 1 : 0;
  }
  if (lane == 0) s_own[warp] = own;
  __syncthreads();
  if (warp == 0) {
    const uint32_t word = __ballot_sync(0xffffffffu, s_own[lane] != 0);
    if (lane == 0) {
      unique[blockIdx.x] = word;
      atomicAdd(&chunk_count[blockIdx.x / (kChunk / kWarps)], __popc(word));
    }
  }
}

// Block: exclusive scan of in[0..count) to out (which may be `in`); returns the total.
__device__ int scan_counts(const int* in, int* out, int count) {
  __shared__ int warp_tot[32];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  int carry = 0;
  for (int base = 0; base < count; base += kChunk) {
    const int v = base + tid < count ? in[base + tid] : 0;
    int incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += y;
    }
    if (lane == 31) warp_tot[warp] = incl;
    __syncthreads();
    int t = warp_tot[lane];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, t, o);
      if (lane >= o) t += y;
    }
    const int before = __shfl_sync(0xffffffffu, t, (warp + 31) & 31), total = __shfl_sync(0xffffffffu, t, 31);
    if (base + tid < count) out[base + tid] = carry + (warp ? before : 0) + incl - v;
    carry += total;
    __syncthreads();
  }
  return carry;
}

// One block per chunk.  The rank of any path c: the unique paths in the chunks before its own (scanned by every block in
// its shared memory, or in place by a launch of its own where that would take several steps), plus those in front of it in
// its chunk (32 words).
constexpr int kMaxChunksShared = 512;
__global__ void __launch_bounds__(kChunk) scan_chunks_kernel(int* chunk_count, int n_chunks, int32_t* num_unique) {
  ss::grid_dependency_enter();
  const int total = scan_counts(chunk_count, chunk_count, n_chunks);
  if (threadIdx.x == 0) *num_unique = total;
}
__global__ void __launch_bounds__(kChunk)
compact_kernel(const int32_t* __restrict__ canon, int n, const uint32_t* __restrict__ unique, const int* chunk_count,
               int n_chunks, const int32_t* __restrict__ slot_in, int32_t* __restrict__ path_to_unique,
               int32_t* __restrict__ unique_paths, int32_t* multiplicity, int32_t* __restrict__ slot_out,
               int32_t* __restrict__ num_unique) {
  ss::grid_dependency_enter();
  __shared__ int s_start[kMaxChunksShared];
  const int tid = threadIdx.x;
  const int* start = chunk_count;
  if (n_chunks <= kMaxChunksShared) {
    const int total = scan_counts(chunk_count, s_start, n_chunks);
    if (blockIdx.x == 0 && tid == 0) *num_unique = total;
    start = s_start;
  }
  const int i = blockIdx.x * kChunk + tid;
  const uint32_t warp_paths = __ballot_sync(0xffffffffu, i < n);
  if (i >= n) return;
  const int c = canon[i], w0 = c / kChunk * (kChunk / 32), w1 = c >> 5;
  int r = start[c / kChunk] + __popc(unique[w1] & ((1u << (c & 31)) - 1u));
  for (int w = w0; w < w1; ++w) r += __popc(unique[w]);
  path_to_unique[i] = r;
  if (c == i) unique_paths[r] = i;
  // (one atomic for the warp's paths that equal its first one, and so on twice: groups of many paths would else be bound by
  //  atomics on one address)
  uint32_t left = warp_paths;
#pragma unroll
  for (int round = 0; round < 2; ++round) {
    const int leader = left ? __ffs(left) - 1 : 0;
    const uint32_t same = __ballot_sync(warp_paths, r == __shfl_sync(warp_paths, r, leader)) & left;
    if (same && (tid & 31) == leader) atomicAdd(&multiplicity[r], __popc(same));
    left &= ~same;
  }
  if ((left >> (tid & 31)) & 1u) atomicAdd(&multiplicity[r], 1);
  if (slot_out) slot_out[i] = slot_in[c];
}

// ---- ss_gather_unique_paths ------------------------------------------------------------------------------------
// One block.  Thread t owns kGatherItems consecutive unique paths per round: it gathers their descriptor rows and the
// block scans the query lengths (thread sums -> warp shuffles -> warp totals -> running carry).
constexpr int kGatherThreads = 1024;
constexpr int kGatherItems = 4;       // (16 per thread - one round for 16384 paths - was measured: 33 -> 60 us, every access 32 sectors wide)

__global__ void __launch_bounds__(kGatherThreads)
gather_unique_kernel(const int32_t* __restrict__ unique_paths, const int32_t* __restrict__ num_unique, int n,
                     const int32_t* __restrict__ path_leaf_node, const int32_t* __restrict__ path_q_len,
                     const int64_t* __restrict__ q_offsets, int32_t* __restrict__ u_leaf, int32_t* __restrict__ u_q_len,
                     int64_t* __restrict__ u_q_offsets, int64_t* __restrict__ u_q_src) {
  ss::grid_dependency_enter();
  __shared__ long long warp_tot[32];
  __shared__ long long carry_s;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int U = min(max(*num_unique, 0), n);
  if (threadIdx.x == 0) { carry_s = 0; u_q_offsets[0] = 0; }
  __syncthreads();
  for (int base = 0; base < n; base += kGatherThreads * kGatherItems) {
    const int p0 = base + threadIdx.x * kGatherItems;
    int len[kGatherItems];
    long long mine = 0;
#pragma unroll
    for (int e = 0; e < kGatherItems; ++e) {
      const int p = p0 + e;
      len[e] = 0;
      if (p < n) {
        int leaf = -1;
        long long src_row = 0;
        if (p < U) {
          const int src = unique_paths[p];
          leaf = path_leaf_node[src];
          len[e] = path_q_len[src];
          src_row = q_offsets[src];
        }
        u_leaf[p] = leaf;
        u_q_len[p] = len[e];
        u_q_src[p] = src_row;
      }
      mine += len[e];
    }
    long long incl = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const long long y = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += y;
    }
    if (lane == 31) warp_tot[warp] = incl;
    __syncthreads();
    if (warp == 0) {
      long long t = warp_tot[lane];
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const long long y = __shfl_up_sync(0xffffffffu, t, o);
        if (lane >= o) t += y;
      }
      warp_tot[lane] = t;
    }
    __syncthreads();
    long long run = carry_s + (warp ? warp_tot[warp - 1] : 0) + incl - mine;   // rows before path p0
#pragma unroll
    for (int e = 0; e < kGatherItems; ++e) {
      run += len[e];
      if (p0 + e < n) u_q_offsets[p0 + e + 1] = run;
    }
    __syncthreads();
    if (threadIdx.x == kGatherThreads - 1) carry_s = run;
    __syncthreads();
  }
}

__global__ void zero_scalar_kernel(int32_t* p) {
  ss::grid_dependency_enter(); *p = 0; }

// Shared memory of small_match_kernel beyond 48 KB, once per device.
static int32_t small_smem_ready() {
  static bool configured[kDeviceSlots] = {false};
  const int slot = current_device_slot();
  if (slot >= 0 && configured[slot]) return SS_OK;
  if (cudaFuncSetAttribute(small_match_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           static_cast<int>(small_match_smem(kSmallMax))) != cudaSuccess ||
      cudaFuncSetAttribute(small_match_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           static_cast<int>(small_match_smem(kSmallMax))) != cudaSuccess) {
    (void)cudaGetLastError();
    return SS_ERR_CUDA;
  }
  if (slot >= 0) configured[slot] = true;
  return SS_OK;
}

struct Layout {
  size_t counters, hash64, table, unique, chunk_count, total;
  uint32_t mask;                                    // table entries - 1
};

static Layout layout(int n) {
  Layout L;
  const size_t m = n > 0 ? n : 1;
  size_t entries = 1;
  while (entries < 2 * m) entries <<= 1;
  L.mask = static_cast<uint32_t>(entries - 1);
  size_t off = 0;
  L.counters = off; off = align_up(off + 64);
  L.hash64 = off; off = align_up(off + m * 8);
  L.table = off; off = align_up(off + (n > kSmallMax ? entries * 8 : 0));
  L.unique = off; off = align_up(off + (m + 31) / 32 * 4);
  L.chunk_count = off; off = align_up(off + (m + kChunk - 1) / kChunk * 4);
  L.total = off;
  return L;
}

}  // namespace dedup
}  // namespace ss

extern "C" int32_t ss_dedup_workspace_bytes(int32_t n_paths, size_t* out_bytes) {
  if (n_paths < 0 || !out_bytes) return SS_ERR_INVALID_ARG;
  *out_bytes = ss::dedup::layout(n_paths).total;
  return SS_OK;
}

extern "C" int32_t ss_dedup_paths(const int32_t* tok_ids, const int64_t* tok_offsets, const int64_t* ctx_key,
                                  const int32_t* slot_in, int32_t n_paths, uint32_t flags, int32_t* canon_out,
                                  int32_t* path_to_unique_out, int32_t* unique_paths_out,
                                  int32_t* multiplicity_out, int32_t* slot_out, int32_t* num_unique_out,
                                  void* workspace, size_t workspace_bytes, void* stream) {
  using namespace ss;
  using namespace ss::dedup;
  if (n_paths < 0 || !num_unique_out) return SS_ERR_INVALID_ARG;
  if (flags & ~SS_FLAG_WEAK_HASH) return SS_ERR_INVALID_ARG;
  cudaStream_t st = as_stream(stream);
  if (n_paths == 0) {
    SS_LAUNCH(zero_scalar_kernel, 1, 1, 0, st, num_unique_out);
    return SS_OK;
  }
  if ((slot_in == nullptr) != (slot_out == nullptr)) return SS_ERR_INVALID_ARG;
  if (!tok_offsets || !canon_out || !path_to_unique_out || !unique_paths_out || !multiplicity_out || !workspace)
    return SS_ERR_INVALID_ARG;
  if (!tok_ids) return SS_ERR_INVALID_ARG;
  if (reinterpret_cast<uintptr_t>(workspace) % kAlign) return SS_ERR_INVALID_ARG;
  const Layout L = layout(n_paths);
  if (workspace_bytes < L.total) return SS_ERR_WORKSPACE_TOO_SMALL;
  char* ws = static_cast<char*>(workspace);
  uint64_t* hash64 = reinterpret_cast<uint64_t*>(ws + L.hash64);
  const int n = n_paths;
  const uint32_t weak = (flags & SS_FLAG_WEAK_HASH) ? 1u : 0u;
  const int hash_blocks = (n + kHashWarps - 1) / kHashWarps, match_blocks = (n + kWarps - 1) / kWarps;
  if (n <= kClusterMax) {
    SS_LAUNCH(cluster_dedup_kernel<false>, kClusterBlocks, kThreads, 0, st, tok_ids, tok_offsets, ctx_key, n, weak, hash64,
              static_cast<uint32_t>(small_table_size(n) - 1), slot_in, canon_out, path_to_unique_out, unique_paths_out,
              multiplicity_out, slot_out, num_unique_out, Gather{}, Selection{});
    return SS_OK;
  }
  if (n <= kSmallMax) {
    unsigned int* arrived = reinterpret_cast<unsigned int*>(ws + L.counters);
    const int32_t rc = small_smem_ready();
    if (rc != SS_OK) return rc;
    SS_LAUNCH(hash_kernel<kAheadSmall>, hash_blocks, kHashWarps * 32, 0, st, tok_ids, tok_offsets, ctx_key, n, weak, hash64,
              static_cast<unsigned long long*>(nullptr), 0u, static_cast<int*>(nullptr), static_cast<int32_t*>(nullptr), arrived);
    SS_LAUNCH(small_match_kernel<false>, match_blocks, kThreads, small_match_smem(n), st, tok_ids, tok_offsets, ctx_key, n, hash64,
              static_cast<uint32_t>(small_table_size(n) - 1), slot_in, canon_out, path_to_unique_out, unique_paths_out,
              multiplicity_out, slot_out, num_unique_out, arrived, Gather{});
    return SS_OK;
  }
  unsigned long long* table = reinterpret_cast<unsigned long long*>(ws + L.table);
  uint32_t* unique = reinterpret_cast<uint32_t*>(ws + L.unique);
  int* chunk_count = reinterpret_cast<int*>(ws + L.chunk_count);
  const int n_chunks = (n + kChunk - 1) / kChunk;
  if (cudaMemsetAsync(table, 0xff, (static_cast<size_t>(L.mask) + 1) * 8, st) != cudaSuccess) {
    (void)cudaGetLastError();
    return SS_ERR_CUDA;
  }
  SS_LAUNCH(hash_kernel<kAheadLarge>, hash_blocks, kHashWarps * 32, 0, st, tok_ids, tok_offsets, ctx_key, n, weak, hash64, table, L.mask,
            chunk_count, multiplicity_out, static_cast<unsigned int*>(nullptr));
  SS_LAUNCH(match_kernel, match_blocks, kThreads, 0, st, tok_ids, tok_offsets, ctx_key, n, hash64, table, L.mask, canon_out,
            unique, chunk_count);
  if (n_chunks > kMaxChunksShared) SS_LAUNCH(scan_chunks_kernel, 1, kChunk, 0, st, chunk_count, n_chunks, num_unique_out);
  SS_LAUNCH(compact_kernel, n_chunks, kChunk, 0, st, canon_out, n, unique, chunk_count, n_chunks, slot_in, path_to_unique_out,
            unique_paths_out, multiplicity_out, slot_out, num_unique_out);
  return SS_OK;
}

// ---------------------------------------------------------------------------------------------------------
// ss_dedup_paths_static: the same deduplication for callers that must not allocate device memory.
//
// Some hosts of this library cannot obtain scratch memory at the moment they need a deduplication pass: a serving
// engine that has already handed all free HBM to its KV-cache pool (an allocation would fail, or shrink the cache),
// a latency-critical scheduling loop in which the device-wide synchronisation hidden in an allocation is not
// acceptable, or a plug-in that is simply not allowed to touch the allocator.  For them the scratch lives in the
// library image itself: a fixed array in device global memory, present on every GPU that loads the library, from
// load until the process ends.
//
// In host code the array's name below is only a handle for the runtime, not a device address; the address that
// kernels can use is obtained once per device with cudaGetSymbolAddress (with that device current) and cached.
// ---------------------------------------------------------------------------------------------------------
namespace ss {
namespace dedup {

constexpr int kStaticMaxPaths = SS_DEDUP_STATIC_MAX_PATHS;
constexpr size_t kStaticScratchBytes = 2u << 20;           // 2 MiB; layout(kStaticMaxPaths).total is about 1.6 MiB
static __device__ __align__(256) unsigned char g_static_scratch[kStaticScratchBytes];

constexpr int kMaxDevices = 64;
static void* g_static_scratch_addr[kMaxDevices] = {nullptr};

// Device address of the scratch array on the current device (looked up on the first call per device).
static int32_t static_scratch_address(void** out) {
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess) { (void)cudaGetLastError(); return SS_ERR_CUDA; }
  if (dev < 0 || dev >= kMaxDevices) return SS_ERR_UNSUPPORTED;
  if (!g_static_scratch_addr[dev]) {
    void* ptr = nullptr;
    if (cudaGetSymbolAddress(&ptr, g_static_scratch) != cudaSuccess || !ptr) {
      (void)cudaGetLastError();
      return SS_ERR_CUDA;
    }
    g_static_scratch_addr[dev] = ptr;
  }
  *out = g_static_scratch_addr[dev];
  return SS_OK;
}

}  // namespace dedup
}  // namespace ss

extern "C" int32_t ss_dedup_paths_static(const int32_t* tok_ids, const int64_t* tok_offsets, const int64_t* ctx_key,
                                         const int32_t* slot_in, int32_t n_paths, uint32_t flags, int32_t* canon_out,
                                         int32_t* path_to_unique_out, int32_t* unique_paths_out,
                                         int32_t* multiplicity_out, int32_t* slot_out, int32_t* num_unique_out,
                                         void* stream) {
  using namespace ss::dedup;
  if (n_paths < 0) return SS_ERR_INVALID_ARG;
  if (n_paths > kStaticMaxPaths) return SS_ERR_UNSUPPORTED;          // larger batches need ss_dedup_paths
  if (layout(n_paths).total > kStaticScratchBytes) return SS_ERR_UNSUPPORTED;
  void* scratch = nullptr;
  const int32_t rc = static_scratch_address(&scratch);
  if (rc != SS_OK) return rc;
  // Nothing in the scratch has to start at zero: what must be clear (the table, counters and counts) is cleared by the
  // call itself.
  return ss_dedup_paths(tok_ids, tok_offsets, ctx_key, slot_in, n_paths, flags, canon_out, path_to_unique_out,
                        unique_paths_out, multiplicity_out, slot_out, num_unique_out, scratch, kStaticScratchBytes,
                        stream);
}

extern "C" int32_t ss_gather_unique_paths(const int32_t* unique_paths, const int32_t* num_unique, int32_t n_paths,
                                          const int32_t* path_leaf_node, const int32_t* path_q_len,
                                          const int64_t* q_offsets, int32_t* u_leaf_out, int32_t* u_q_len_out,
                                          int64_t* u_q_offsets_out, int64_t* u_q_src_out, void* stream) {
  using namespace ss;
  using namespace ss::dedup;
  if (n_paths < 0 || !u_q_offsets_out) return SS_ERR_INVALID_ARG;
  cudaStream_t st = as_stream(stream);
  if (n_paths == 0) {
    if (cudaMemsetAsync(u_q_offsets_out, 0, sizeof(int64_t), st) != cudaSuccess) {
      (void)cudaGetLastError();
      return SS_ERR_CUDA;
    }
    return SS_OK;
  }
  if (!unique_paths || !num_unique || !path_leaf_node || !path_q_len || !q_offsets || !u_leaf_out || !u_q_len_out ||
      !u_q_src_out)
    return SS_ERR_INVALID_ARG;
  SS_LAUNCH(gather_unique_kernel, 1, kGatherThreads, 0, st, unique_paths, num_unique, n_paths, path_leaf_node, path_q_len,
            q_offsets, u_leaf_out, u_q_len_out, u_q_offsets_out, u_q_src_out);
  return SS_OK;
}

// ---- ss_candidate_step ------------------------------------------------------------------------------------------------
namespace ss {
namespace dedup {

// The front of a step of up to kSmallMax paths - deduplication, gather, selection - in one launch (a cluster, the selection's
// blocks beside it) or two (the selection's blocks beside the hash, the gather by the block that compacts) where the four calls
// take three or four.  Measured, the step: 8 paths 33.8 -> 29.3 us, 1024 paths 104.8 -> 94.7 (two levels 183.4 -> 174.2), 8
// verification paths 40.2 -> 36.5.  Part of it (1024 paths) are the loads of the hash, eight a lane in flight instead of one.
static int32_t launch_front(const ss_device_step_t& s, cudaStream_t st) {
  const Layout L = layout(s.n_paths);
  char* ws = static_cast<char*>(s.dedup_workspace);
  uint64_t* hash64 = reinterpret_cast<uint64_t*>(ws + L.hash64);
  const int n = s.n_paths;
  const uint32_t weak = (s.dedup_flags & SS_FLAG_WEAK_HASH) ? 1u : 0u, mask = static_cast<uint32_t>(small_table_size(n) - 1);
  const Gather G{s.path_leaf_node, s.path_q_len, s.q_offsets, s.u_leaf, s.u_q_len, s.u_q_offsets, s.u_q_src};
  const Selection T{s.scores, s.seg_offsets, s.n_segments, s.top_k, s.survivors, s.keep,
                    reinterpret_cast<uint64_t*>(static_cast<char*>(s.topk_workspace) + kAlign), static_cast<int32_t*>(s.topk_workspace)};
  if (n <= kClusterMax) {
    const int clusters = 1 + (s.n_segments + kClusterBlocks - 1) / kClusterBlocks;
    SS_LAUNCH(cluster_dedup_kernel<true>, clusters * kClusterBlocks, kThreads, 0, st, s.tok_ids, s.tok_offsets, s.ctx_key, n, weak, hash64,
              mask, s.slot_in, s.canon, s.path_to_unique, s.unique_paths, s.multiplicity, s.slot_out, s.num_unique, G, T);
    return SS_OK;
  }
  const int32_t rc = small_smem_ready();
  if (rc != SS_OK) return rc;
  const int hash_blocks = (n + kHashWarps - 1) / kHashWarps, match_blocks = (n + kWarps - 1) / kWarps;
  unsigned int* arrived = reinterpret_cast<unsigned int*>(ws + L.counters);
  SS_LAUNCH(hash_select_kernel, hash_blocks + s.n_segments, kHashWarps * 32, 0, st, s.tok_ids, s.tok_offsets, s.ctx_key, n, weak, hash64,
            arrived, hash_blocks, T);
  SS_LAUNCH(small_match_kernel<true>, match_blocks, kThreads, small_match_smem(n), st, s.tok_ids, s.tok_offsets, s.ctx_key, n, hash64, mask,
            s.slot_in, s.canon, s.path_to_unique, s.unique_paths, s.multiplicity, s.slot_out, s.num_unique, arrived, G);
  return SS_OK;
}

// True if the deduplication, the gather and the selection would accept their arguments.  (The attention looks at its own behind them,
// as where the four calls are made one after the other; the selection's results are then there already.)
static bool front_args_ok(const ss_device_step_t& s) {
  if ((s.slot_in == nullptr) != (s.slot_out == nullptr) || s.top_k < 1 || (s.dedup_flags & ~SS_FLAG_WEAK_HASH)) return false;
  const void* const needed[] = {s.tok_ids, s.tok_offsets, s.canon, s.path_to_unique, s.unique_paths, s.multiplicity, s.num_unique,
                                s.dedup_workspace, s.path_leaf_node, s.path_q_len, s.q_offsets, s.u_leaf, s.u_q_len, s.u_q_offsets,
                                s.u_q_src, s.scores, s.seg_offsets, s.survivors, s.keep, s.topk_workspace};
  for (const void* p : needed)
    if (!p) return false;
  size_t topk_bytes = 0;
  if (ss_topk_workspace_bytes(s.n_paths, &topk_bytes) != SS_OK) return false;
  return reinterpret_cast<uintptr_t>(s.dedup_workspace) % kAlign == 0 && reinterpret_cast<uintptr_t>(s.topk_workspace) % kAlign == 0 &&
         s.dedup_workspace_bytes >= layout(s.n_paths).total && s.topk_workspace_bytes >= topk_bytes;
}

}  // namespace dedup
}  // namespace ss

int32_t ss::candidate_step(const ss_device_step_t& s, void* stream, cudaEvent_t q_ready, bool out_on_host) {
  using namespace ss::dedup;
  const int n = s.n_paths;
  // The selection shares the front's launches where 256 threads (1024 in the cluster form) are as many as its own launch would
  // take, and its segments are not many times the other blocks.
  const bool front = n > 0 && n <= kSmallMax && s.n_segments > 0 && s.n_segments <= 1024 && front_args_ok(s) &&
                     (n <= kClusterMax || topk::block_threads(n, s.n_segments) <= kHashWarps * 32);
  int32_t rc;
  if (front) {
    rc = launch_front(s, as_stream(stream));
    return rc != SS_OK ? rc : attn::tree_attention(s.attn, s.attn_workspace, s.attn_workspace_bytes, stream, q_ready, out_on_host);
  }
  rc = ss_dedup_paths(s.tok_ids, s.tok_offsets, s.ctx_key, s.slot_in, n, s.dedup_flags, s.canon, s.path_to_unique, s.unique_paths,
                      s.multiplicity, s.slot_out, s.num_unique, s.dedup_workspace, s.dedup_workspace_bytes, stream);
  if (rc != SS_OK) return rc;
  rc = ss_gather_unique_paths(s.unique_paths, s.num_unique, n, s.path_leaf_node, s.path_q_len, s.q_offsets, s.u_leaf, s.u_q_len,
                              s.u_q_offsets, s.u_q_src, stream);
  if (rc != SS_OK) return rc;
  rc = attn::tree_attention(s.attn, s.attn_workspace, s.attn_workspace_bytes, stream, q_ready, out_on_host);
  if (rc != SS_OK) return rc;
  return ss_topk_prune(s.scores, s.seg_offsets, s.n_segments, n, s.top_k, s.survivors, s.keep, s.topk_workspace, s.topk_workspace_bytes,
                       stream);
}

extern "C" int32_t ss_candidate_step(const ss_device_step_t* step, void* stream) {
  if (!step || step->struct_size != sizeof(ss_device_step_t) || !step->attn) return SS_ERR_INVALID_ARG;
  return ss::candidate_step(*step, stream, nullptr, false);
}
