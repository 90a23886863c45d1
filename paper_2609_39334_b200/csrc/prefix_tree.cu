// ss_build_prefix_tree: radix tree of candidate paths over whole KV pages, from raw token ids (paper, Section
// "Computation Deduplication": candidates of a step share a large part of their tokens; Section "Experimental Setup":
// prefix KV caching and sharing).  Only whole pages are shared; every path gets a private leaf node.
//
// ONE launch whose phases are separated by a barrier over all its blocks: one block, a cluster of 8, or one block per SM
// (a cooperative launch).  No token is hashed and none that is known to be shared is read twice.
//
//   sort    The paths are sorted by refinement (a multikey quicksort with longest common prefixes as keys).  All
//           positions start in one group; round 0 sorts by the first token.  In a round every group of two or more picks one
//           of its paths as the pivot, and every other member compares itself with it, from the length that the group is known
//           to share: a warp per path, streaming both.  Its key - below or above the pivot, common length, first differing token - sorts the group;
//           members with equal keys share that many tokens plus one, and make a group of the next round.  Members that equal
//           the pivot, or that end where they differ from it, are settled.  Neighbours that were told apart in a round share
//           exactly the smaller of their two lengths, so the common prefixes of the sorted neighbours, which the tree is made
//           of, come out of the keys.  A round settles at least the pivots; the pivot is picked pseudo-randomly, so the number
//           of rounds is that of a quicksort's levels in the worst case and the depth of the tree in ordinary ones (3 or 4).
//             compare   a warp per position: boundaries of the groups from the last round's sorted keys (32-ary search), then
//                       the new key; a group of up to 8 that has met a pivot is finished at once, every member
//                       against every other (its rank is the number below it, what it shares with the rank before the
//                       most that it shares with any of them)
//             ranks     a warp per position counts the smaller keys of its group; with groups of more than 256 a block per
//                       1024 positions sorts (group, key, position), then the sorted runs are merged by ranks, 4 at a time: a lane
//                       per position and run counts the keys in front by binary search
//   tree    Inner nodes are the intervals of neighbours that share more pages than their surroundings (the LCP-interval
//           tree).  A warp per position finds its interval with nearest-smaller-value searches of 32 entries a step, over
//           the entries and over their minima by 32; depth-first numbering (leaves included) comes from a prefix sum of
//           the intervals per start rank; parents follow from the neighbours of an interval.
//
// Bound: HBM, one pass over the shared prefixes (268 MB for 16384 paths with prompts of 4096 tokens, 41 us), and for small
// inputs the latency of a dozen dependent phases.  Measured: 16384 paths / 76 M ids 149 us (of which 61 the pass over the
// prompts; page hashes, a bitonic sort with a string comparator and a pass over the neighbours: 1729), 64 paths 25 us (135).
#include "common.cuh"

namespace ss {
namespace ptree {

constexpr int kThreads = 1024;
constexpr int kWarps = kThreads / 32;
constexpr int kTile = 1024;                       // positions that are sorted in shared memory together (16384 paths: 1024 151
                                                  // us, 512 159, 256 173; below a few thousand 2 to 4 us less with 256)
constexpr int kUnroll = 8;                        // 128-byte loads in flight per warp and path (16384 paths: 8 151 us, 16 148;
                                                  // 512 paths 46.8 and 48.1)
constexpr int kPairs = 8;                         // a group of up to this many is finished with all pairs: 7 comparisons in a
                                                  // row (9 us) against two or three more rounds (8 us each)
constexpr int kCount = 256;                       // ranks by counting up to this group size: 8 keys a lane (1.2 us) against a
                                                  // tile sort (13 us); beyond, counting grows with the square
constexpr int kFan = 4;                           // sorted runs merged in a pass.  1M paths of 6 tokens: all 1024 tiles at once 34.4 ms
                                                  // (a search in every tile for every position), 4 2.3, 8 2.6, 2 2.4; 64000 paths 344 us,
                                                  // 225, 229, 236; 16384 (16 tiles) 145 at once, 145, 143, 152
constexpr uint32_t kInf = 0x7fffffffu;            // "common length" of a path with itself
constexpr unsigned long long kBarrierLimitNs = 4000000000ull;

struct Args {
  const int32_t* tok_ids;
  const int64_t* tok_offsets;
  int n, page, n_tiles;
  int32_t* status;               // first word of the workspace
  unsigned int* arrived;         // grid barrier
  unsigned int* flags;           // [4]: what the round's groups need (kMore, kBig), rounds in turn
  uint64_t* key[2];
  int* perm[2];
  int *gs, *ge;                  // per position: its group [gs, ge)
  int* lcp;                      // per rank: pages shared with the rank before
  int *bmin, *c_start, *c_end, *outer, *cnt, *block_sum;
  int32_t *order, *path_leaf_node, *node_parent, *node_kv_len, *node_src_path, *node_src_offset, *num_nodes;
};
constexpr unsigned int kMore = 1, kBig = 2, kMixed = 4;
constexpr int kCleared = 256;                     // bytes from the status word on: it, the barrier, the flags

// ---- barrier over all blocks ----------------------------------------------------------------------------------------
// False when the wait ran out (status SS_ERR_TIMEOUT; every block leaves).  A grid that is one cluster uses the hardware's
// barrier (0.3 us against 1.5 us).
template <bool CLUSTER>
__device__ __forceinline__ bool grid_barrier(const Args& A, unsigned int& target) {
  if (CLUSTER) {
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
    return true;
  }
  __shared__ int ok;
  __syncthreads();
  target += gridDim.x;
  if (threadIdx.x == 0) {
    __threadfence();
    atomicAdd(A.arrived, 1u);
    unsigned long long t0, t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t0));
    ok = 1;
    for (;;) {
      unsigned int v;
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(A.arrived) : "memory");
      if (static_cast<int>(v - target) >= 0) break;
      asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
      if (t - t0 > kBarrierLimitNs) { set_status(A.status, SS_ERR_TIMEOUT); ok = 0; break; }
    }
    __threadfence();
  }
  __syncthreads();
  return ok != 0;
}

// ---- sort -------------------------------------------------------------------------------------------------------------
__device__ __forceinline__ uint32_t ordered(int32_t token) { return static_cast<uint32_t>(token) ^ 0x80000000u; }
// Common length that a key stands for (see make_key).
__device__ __forceinline__ uint32_t key_len(uint64_t k) {
  const uint32_t f = static_cast<uint32_t>(k >> 32) & kInf;
  return (k >> 63) ? kInf - f : f;
}
// All paths with this key are equal: the pivot's own, or paths that end where they differ from it.
__device__ __forceinline__ bool key_settled(uint64_t k) { return !(k >> 63) && static_cast<uint32_t>(k) == 0; }

// Whole warp: what paths `me` and `other` share (they are known to share `base` tokens) and which comes first by tokens, a
// proper prefix first.
struct Order {
  int len, sign;               // sign < 0: `me` before `other`; 0: equal
  bool ends;                   // `me` ends at len
  uint32_t token;              // of `me` at len (if it does not end there), in the order of its bits
};
__device__ Order compare_paths(const Args& A, int me, int other, int base, int lane) {
  const int64_t a0 = A.tok_offsets[me], b0 = A.tok_offsets[other];
  const int la = static_cast<int>(A.tok_offsets[me + 1] - a0), lb = static_cast<int>(A.tok_offsets[other + 1] - b0);
  const int m = min(la, lb);
  const int32_t *a = A.tok_ids + a0, *b = A.tok_ids + b0;
  int l = m;
  // 32 tokens first (most pairs differ at once or not for long), then kUnroll * 32 a step
  int32_t x0 = base + lane < m ? __ldg(a + base + lane) : 0, y0 = base + lane < m ? __ldg(b + base + lane) : 0;
  int at = base;                                              // x0, y0 are the tokens at `at` + lane
  uint32_t bal = __ballot_sync(0xffffffffu, x0 != y0);
  if (bal) {
    l = base + __ffs(bal) - 1;
  } else {
    for (int t0 = base + 32; t0 < m; t0 += 32 * kUnroll) {
      int32_t x[kUnroll], y[kUnroll];
#pragma unroll
      for (int u = 0; u < kUnroll; ++u) {
        const int t1 = t0 + 32 * u + lane;
        x[u] = t1 < m ? __ldg(a + t1) : 0;
        y[u] = t1 < m ? __ldg(b + t1) : 0;
      }
      int first = 32 * kUnroll;
#pragma unroll
      for (int u = kUnroll - 1; u >= 0; --u)
        if (x[u] != y[u]) { first = 32 * u + lane; x0 = x[u]; y0 = y[u]; }
      const int found = __reduce_min_sync(0xffffffffu, first);
      if (found < 32 * kUnroll) { l = t0 + found; at = l - (found & 31); break; }
    }
  }
  Order o;
  o.len = l;
  o.ends = l == la;
  if (l == m) {
    o.sign = la < lb ? -1 : (la > lb ? 1 : 0);
    o.token = o.ends ? 0 : ordered(__ldg(a + l));
  } else {
    o.token = ordered(__shfl_sync(0xffffffffu, x0, l - at));
    o.sign = o.token < ordered(__shfl_sync(0xffffffffu, y0, l - at)) ? -1 : 1;
  }
  return o;
}

// The key of a path against the pivot, ascending in the paths' order:
//   below the pivot  0 | l | token + 1, or 0 if the path ends at l    (shorter common prefix = smaller path)
//   equal to it      0 | kInf | 0
//   above it         1 | kInf - l | token
__device__ __forceinline__ uint64_t make_key(const Order& o) {
  if (o.sign == 0) return static_cast<uint64_t>(kInf) << 32;
  if (o.sign < 0) return (static_cast<uint64_t>(o.len) << 32) | (o.ends ? 0u : o.token + 1);
  return (1ull << 63) | (static_cast<uint64_t>(kInf - o.len) << 32) | o.token;
}

// Whole warp: number of keys in the ascending k[0..len) that are below `key` (OR_EQUAL: not above it).
template <bool OR_EQUAL>
__device__ __forceinline__ int count_below(const uint64_t* k, int len, uint64_t key, int lane) {
  int lo = 0;
  while (len > 32) {
    const int step = (len + 31) >> 5, i = lane * step;
    const uint64_t v = i < len ? k[lo + i] : ~0ull;
    const int c = __popc(__ballot_sync(0xffffffffu, i < len && (OR_EQUAL ? v <= key : v < key)));
    if (c == 0) return lo;
    const int at = (c - 1) * step + 1;                        // k[lo + at - 1] is below
    len = min(step - 1, len - at);
    lo += at;
  }
  const uint64_t v = lane < len ? k[lo + lane] : ~0ull;
  return lo + __popc(__ballot_sync(0xffffffffu, lane < len && (OR_EQUAL ? v <= key : v < key)));
}

// Sorts the positions of kThreads / kTile tiles, each by (group, key, position): keys and paths of the round, kin / pin ->
// kout / pout.  An entry per thread; partners in the warp through shuffles, the others through shared memory.
__device__ void sort_tiles(const Args& A, int first_tile, const uint64_t* kin, const int* pin, uint64_t* kout, int* pout) {
  __shared__ uint64_t s_key[kThreads];
  __shared__ uint32_t s_at[kThreads];
  const int tid = threadIdx.x % kTile, at0 = threadIdx.x - tid;   // position in the tile, the tile's place in shared memory
  const int p0 = (first_tile + threadIdx.x / kTile) * kTile, count = min(kTile, A.n - p0);
  uint64_t k = ~0ull;
  uint32_t at = 0xffffffffu;                                  // first position of the group in the tile << 16 | position
  bool open = false;
  if (tid < count) {
    const int g = A.gs[p0 + tid];
    open = A.ge[p0 + tid] - g > 1;
    k = open ? kin[p0 + tid] : 0;
    at = (static_cast<uint32_t>(max(g - p0, 0)) << 16) | static_cast<uint32_t>(tid);
  }
  if (!__syncthreads_or(open)) return;
  int n_pad = 2;                                              // (of the block's first tile, the fullest)
  while (n_pad < min(kTile, A.n - first_tile * kTile)) n_pad <<= 1;
  for (int size = 2; size <= n_pad; size <<= 1) {
    for (int stride = size >> 1; stride > 0; stride >>= 1) {
      uint64_t kb;
      uint32_t ab;
      if (stride >= 32) {
        s_key[at0 + tid] = k;
        s_at[at0 + tid] = at;
        __syncthreads();
        kb = s_key[at0 + (tid ^ stride)];
        ab = s_at[at0 + (tid ^ stride)];
        __syncthreads();
      } else {
        kb = __shfl_xor_sync(0xffffffffu, k, stride);
        ab = __shfl_xor_sync(0xffffffffu, at, stride);
      }
      const uint32_t ga = at >> 16, gb = ab >> 16;
      const bool above = ga != gb ? ga > gb : (k != kb ? k > kb : at > ab);
      const bool keep_low = ((tid & stride) == 0) == ((tid & size) == 0);
      if (above == keep_low) { k = kb; at = ab; }
    }
  }
  if (tid < count) {
    kout[p0 + tid] = k;
    pout[p0 + tid] = pin[p0 + static_cast<int>(at & 0xffffu)];
  }
}

// ---- tree -------------------------------------------------------------------------------------------------------------
// Inner nodes are the LCP intervals of lcp[]: maximal runs of ranks a..b whose neighbours all share at least d pages
// (lcp[a+1..b] >= d, with equality somewhere) while lcp[a] < d and lcp[b+1] < d (lcp[n] counts as 0).  The interval is
// created by its first position x with lcp[x] == d.
//
// Whole warp: largest p < x with lcp[p] < bound (STRICT) or <= bound; lcp[0] = 0 ends every search for bound >= 0 (> 0 if
// strict).
template <bool STRICT>
__device__ int prev_below(const Args& A, int x, int bound, int lane) {
  auto hit = [&](int val) { return STRICT ? val < bound : val <= bound; };
  const int blk = x >> 5;
  {
    const int p = (blk << 5) + lane;
    const uint32_t b = __ballot_sync(0xffffffffu, p < x && hit(A.lcp[p < x ? p : 0]));
    if (b) return (blk << 5) + 31 - __clz(b);
  }
  for (int top = blk; top > 0; top -= 32) {                   // blocks top-32 .. top-1
    const int q = top - 32 + lane;
    const uint32_t b = __ballot_sync(0xffffffffu, q >= 0 && hit(A.bmin[q >= 0 ? q : 0]));
    if (!b) continue;
    const int found = top - 32 + 31 - __clz(b);
    const uint32_t c = __ballot_sync(0xffffffffu, hit(A.lcp[(found << 5) + lane]));
    return (found << 5) + 31 - __clz(c);
  }
  return 0;
}
// Whole warp: smallest q > x with lcp[q] < bound (STRICT) or <= bound; n if there is none.
template <bool STRICT>
__device__ int next_below(const Args& A, int x, int bound, int lane) {
  auto hit = [&](int val) { return STRICT ? val < bound : val <= bound; };
  const int n = A.n, blk = x >> 5, n_blk = (n + 31) >> 5;
  {
    const int q = (blk << 5) + lane;
    const uint32_t b = __ballot_sync(0xffffffffu, q > x && q < n && hit(A.lcp[q < n ? q : 0]));
    if (b) return (blk << 5) + __ffs(b) - 1;
  }
  for (int low = blk + 1; low < n_blk; low += 32) {
    const int q = low + lane;
    const uint32_t b = __ballot_sync(0xffffffffu, q < n_blk && hit(A.bmin[q < n_blk ? q : 0]));
    if (!b) continue;
    const int found = low + __ffs(b) - 1, at = (found << 5) + lane;
    const uint32_t c = __ballot_sync(0xffffffffu, at < n && hit(A.lcp[at < n ? at : 0]));
    return (found << 5) + __ffs(c) - 1;
  }
  return n;
}
// Creating position of the interval of depth d that contains position pos (lcp[pos] >= d, d > 0).
__device__ __forceinline__ int creator_of(const Args& A, int pos, int d, int lane) {
  return next_below<false>(A, prev_below<true>(A, pos, d, lane), d, lane);
}

// Block: exclusive scan of a[lo..hi) in place, starting from `carry`.
__device__ void scan_range(int* a, int lo, int hi, int carry) {
  __shared__ int warp_tot[kWarps];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int base = lo; base < hi; base += kThreads) {
    const int i = base + threadIdx.x, v = i < hi ? a[i] : 0;
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
    if (i < hi) a[i] = carry + (warp ? before : 0) + incl - v;
    carry += total;
    __syncthreads();
  }
}

template <bool CLUSTER>
__device__ __forceinline__ void build(const Args& A) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int n = A.n, n_warps = gridDim.x * kWarps, wid = blockIdx.x * kWarps + warp;
  unsigned int target = 0;
  if (blockIdx.x == 0 && threadIdx.x == 0) *A.num_nodes = 0;
  if (CLUSTER) {                                              // (in a grid it is cleared in front of the launch: a launch of its own costs 64
    if (blockIdx.x == 0 && threadIdx.x < kCleared / 4) A.status[threadIdx.x] = 0;   // paths 2 us)
    asm volatile("barrier.cluster.arrive.release;" ::: "memory");
  }

  // ---- sort: round 0 has one group of all positions, in index order ---------------------------------------------------
  int kc = 0, pc = 0;                                         // buffers of the sorted keys and the paths
  for (unsigned int round = 0;; ++round) {
    const uint64_t* ks = A.key[kc];
    unsigned int need = 0;
    if (round == 0) {
      // Against the empty path: the key is the first token (a warp that compares two long paths of one problem would hold
      // up all others).  If all of them begin alike there is nothing to sort.
      auto first_key = [&](int i) {
        const int64_t o = A.tok_offsets[i];
        return make_key(A.tok_offsets[i + 1] > o ? Order{0, 1, false, ordered(__ldg(A.tok_ids + o))} : Order{0, 0, true, 0});
      };
      const uint64_t key0 = first_key(0);
      for (int p = blockIdx.x * kThreads + threadIdx.x; p < n; p += gridDim.x * kThreads) {
        const uint64_t k = first_key(p);
        A.key[0][p] = A.key[1][p] = k;
        A.perm[pc][p] = p;
        A.gs[p] = 0;
        A.ge[p] = n;
        if (p == 0) A.lcp[0] = 0;
        if (n == 1) A.order[0] = 0;
        else need |= kMore | (n > kCount ? kBig : 0) | (k != key0 ? kMixed : 0);
      }
      need = __reduce_or_sync(0xffffffffu, need);
    }
    for (int p = wid; round > 0 && p < n; p += n_warps) {
      int g = A.gs[p], e = A.ge[p], base, me;
      if (e - g == 1) continue;                                // settled
      {
        me = A.perm[pc][p];
        const uint64_t k = ks[p];
        const int g1 = g + count_below<false>(ks + g, e - g, k, lane), e1 = g + count_below<true>(ks + g, e - g, k, lane);
        const int m = e1 - g1;
        if (lane == 0 && p == g1 && p > g) A.lcp[p] = static_cast<int>(min(key_len(ks[p - 1]), key_len(k))) / A.page;
        base = static_cast<int>(key_len(k)) + 1;
        const bool equal = key_settled(k), pairs = !equal && (m == 1 || (m <= kPairs && round > 1));
        int rank = p - g1, shared = 0;                         // in the group; tokens shared with the rank before
        if (equal) {
          shared = static_cast<int>(A.tok_offsets[me + 1] - A.tok_offsets[me]);
        } else if (pairs) {
          rank = 0;
          for (int x = 0; x < m; ++x) {
            if (g1 + x == p) continue;
            const Order o = compare_paths(A, me, A.perm[pc][g1 + x], base, lane);
            if (o.sign > 0 || (o.sign == 0 && g1 + x < p)) {
              ++rank;
              shared = max(shared, o.len);
            }
          }
        }
        if (equal || pairs) {
          if (lane == 0) {
            A.order[g1 + rank] = me;
            if (rank > 0) A.lcp[g1 + rank] = shared / A.page;
            A.gs[p] = p;
            A.ge[p] = p + 1;
          }
          continue;
        }
        if (lane == 0) {
          A.gs[p] = g1;
          A.ge[p] = e1;
        }
        g = g1;
        e = e1;
      }
      const int m = e - g;
      need |= kMore | (m > kCount ? kBig : 0);
      uint32_t r = (static_cast<uint32_t>(g) * 0x9e3779b1u) ^ ((round + 1) * 0x85ebca6bu);
      r = (r ^ (r >> 15)) * 0x2c1b3c6du;
      const int at = g + static_cast<int>((r >> 3) % static_cast<uint32_t>(m));
      const int pivot = A.perm[pc][at];
      Order o{0, 0, false, 0};
      if (me != pivot) o = compare_paths(A, me, pivot, base, lane);
      if (lane == 0) A.key[kc ^ 1][p] = make_key(o);
    }
    if (CLUSTER && round == 0) asm volatile("barrier.cluster.wait.acquire;" ::: "memory");   // (the flags are clear)
    if (lane == 0 && need) atomicOr(&A.flags[round & 3], need);
    if (!grid_barrier<CLUSTER>(A, target)) return;
    const unsigned int flags = *reinterpret_cast<volatile unsigned int*>(&A.flags[round & 3]);
    if (!(flags & kMore)) break;
    if (blockIdx.x == 0 && threadIdx.x == 0) A.flags[(round + 2) & 3] = 0;
    if (round == 0 && !(flags & kMixed)) continue;
    if (!(flags & kBig)) {
      const uint64_t* kn = A.key[kc ^ 1];
      for (int p = wid; p < n; p += n_warps) {
        const int g = A.gs[p], e = A.ge[p];
        if (e - g == 1) continue;
        const uint64_t k = kn[p];
        int below = 0;
        for (int q = g + lane; q < e; q += 32) below += kn[q] < k || (kn[q] == k && q < p) ? 1 : 0;
        below = static_cast<int>(__reduce_add_sync(0xffffffffu, static_cast<unsigned int>(below)));
        if (lane == 0) {
          A.key[kc][g + below] = k;
          A.perm[pc ^ 1][g + below] = A.perm[pc][p];
        }
      }
      pc ^= 1;
      if (!grid_barrier<CLUSTER>(A, target)) return;
      continue;
    }
    for (int t = blockIdx.x * (kThreads / kTile); t < A.n_tiles; t += gridDim.x * (kThreads / kTile))
      sort_tiles(A, t, A.key[kc ^ 1], A.perm[pc], A.key[kc], A.perm[pc ^ 1]);
    if (!grid_barrier<CLUSTER>(A, target)) return;
    // Sorted runs of `span` positions are merged, kFan at a time: a lane for each run that may hold keys of the position's group.
    pc ^= 1;
    for (int span = kTile; span < n; span *= kFan) {
      const int sub = lane & (kFan - 1);
      for (int p0 = wid * (32 / kFan); p0 < n; p0 += n_warps * (32 / kFan)) {
        const int p = p0 + lane / kFan;
        int g = 0, e = 0, rank = 0, first = 0;
        uint64_t k = 0;
        if (p < n) {
          g = A.gs[p];
          e = A.ge[p];
        }
        if (e - g > 1) {
          const int run = p / span, other = run / kFan * kFan + sub;
          first = max(g, run / kFan * kFan * span);
          k = A.key[kc][p];
          if (other == run) {
            rank = p - max(g, run * span);
          } else if (other * span < e && (other + 1) * span > g) {
            const int begin = max(g, other * span);
            int lo = begin, hi = min(e, (other + 1) * span);   // first position that does not come before p
            while (lo < hi) {
              const int mid = (lo + hi) >> 1;
              const uint64_t v = A.key[kc][mid];
              if (other < run ? v <= k : v < k) lo = mid + 1; else hi = mid;
            }
            rank = lo - begin;
          }
        }
        __syncwarp();
#pragma unroll
        for (int o = kFan >> 1; o > 0; o >>= 1) rank += __shfl_xor_sync(0xffffffffu, rank, o);
        if (sub == 0 && e - g > 1) {
          A.key[kc ^ 1][first + rank] = k;
          A.perm[pc ^ 1][first + rank] = A.perm[pc][p];
        }
      }
      kc ^= 1;
      pc ^= 1;
      if (!grid_barrier<CLUSTER>(A, target)) return;
    }
  }
  const int* path_of = A.order;

  // ---- tree -----------------------------------------------------------------------------------------------------------
  for (int p0 = wid * 32; p0 <= n; p0 += n_warps * 32) {
    const int p = p0 + lane;
    if (p <= n) A.cnt[p] = 0;
    const int m = __reduce_min_sync(0xffffffffu, p < n ? A.lcp[p] : 0x7fffffff);
    if (lane == 0 && p0 < n) A.bmin[p0 >> 5] = m;
  }
  if (!grid_barrier<CLUSTER>(A, target)) return;
  // intervals: creating positions, start and end ranks, number per start rank, intervals around it with the same start
  for (int x = wid; x < n; x += n_warps) {
    const int d = A.lcp[x];
    int start = -1, end = 0, outer = 0;
    if (x > 0 && d > 0) {
      const int p = prev_below<false>(A, x, d, lane);
      const int left = A.lcp[p];
      if (left < d) {                                          // no earlier position of this interval has depth d
        start = p;
        end = next_below<true>(A, x, d, lane) - 1;
        for (int e = end;;) {                                  // outwards
          const int v = e + 1 < n ? A.lcp[e + 1] : 0;
          if (v <= left) break;
          ++outer;
          e = next_below<true>(A, e + 1, v, lane) - 1;
        }
      }
    }
    if (lane == 0) {
      A.c_start[x] = start;
      A.c_end[x] = end;
      A.outer[x] = outer;
      if (start >= 0) atomicAdd(&A.cnt[start], 1);
    }
  }
  if (!grid_barrier<CLUSTER>(A, target)) return;
  // cnt[a] (intervals that start at rank a) -> exclusive prefix sums; cnt[n] = number of inner nodes
  {
    const int per = (n + static_cast<int>(gridDim.x)) / static_cast<int>(gridDim.x);
    const int lo = min(static_cast<int>(blockIdx.x) * per, n + 1), hi = min(lo + per, n + 1);
    int carry = 0;
    if (gridDim.x > 1) {
      __shared__ int tot[kWarps];
      int sum = 0;
      for (int i = lo + threadIdx.x; i < hi; i += kThreads) sum += A.cnt[i];
      sum = static_cast<int>(__reduce_add_sync(0xffffffffu, static_cast<unsigned int>(sum)));
      if (lane == 0) tot[warp] = sum;
      __syncthreads();
      if (warp == 0) {
        sum = static_cast<int>(__reduce_add_sync(0xffffffffu, static_cast<unsigned int>(tot[lane])));
        if (lane == 0) A.block_sum[blockIdx.x] = sum;
      }
      if (!grid_barrier<CLUSTER>(A, target)) return;
      for (int i = lane; i < static_cast<int>(blockIdx.x); i += 32) carry += A.block_sum[i];
      carry = static_cast<int>(__reduce_add_sync(0xffffffffu, static_cast<unsigned int>(carry)));
    }
    scan_range(A.cnt, lo, hi, carry);
  }
  if (!grid_barrier<CLUSTER>(A, target)) return;
  if (blockIdx.x == 0 && threadIdx.x == 0) *A.num_nodes = n + A.cnt[n];   // (cnt[n] had no interval: it is the total)
  // Nodes.  The depth-first rank of an interval among the inner nodes: intervals that start earlier come first, and of
  // those that start at the same rank the outer ones.  (d pages deep <=> d * page tokens on the chain above.)
  auto inner_id = [&](int x) { return A.cnt[A.c_start[x]] + A.outer[x] + A.c_start[x]; };   // (`start` leaves precede it)
  for (int r = wid; r < n; r += n_warps) {
    const int depth = A.lcp[r], right1 = r + 1 < n ? A.lcp[r + 1] : 0;
    const int a = A.c_start[r];
    if (a >= 0) {                                              // the interval created at this position
      const int e = A.c_end[r], left = A.lcp[a], right = e + 1 < n ? A.lcp[e + 1] : 0;
      const int id = inner_id(r);
      int parent = -1, pd = 0;
      if (right > left) {                                      // the next outer interval starts at the same rank
        parent = id - 1;
        pd = right;
      } else if (left > 0) {
        parent = inner_id(creator_of(A, a, left, lane));
        pd = left;
      }
      if (lane == 0) {
        A.node_parent[id] = parent;
        A.node_kv_len[id] = (depth - pd) * A.page;
        A.node_src_path[id] = path_of[a];
        A.node_src_offset[id] = pd * A.page;
      }
    }
    const int pd = max(depth, right1);                         // the leaf of rank r
    int parent = -1;
    if (pd > 0) parent = inner_id(creator_of(A, depth >= right1 ? r : r + 1, pd, lane));
    if (lane == 0) {
      const int path = path_of[r], id = r + A.cnt[r + 1];      // every interval that starts at a rank <= r precedes it
      A.node_parent[id] = parent;
      A.node_kv_len[id] = static_cast<int>(A.tok_offsets[path + 1] - A.tok_offsets[path]) - pd * A.page;
      A.node_src_path[id] = path;
      A.node_src_offset[id] = pd * A.page;
      A.path_leaf_node[r] = id;
    }
  }
}

__global__ void __launch_bounds__(kThreads, 1) prefix_tree_grid_kernel(const __grid_constant__ Args A) {
  ss::grid_dependency_enter();
  build<false>(A);
}
__global__ void __launch_bounds__(kThreads, 1) prefix_tree_cluster_kernel(const __grid_constant__ Args A) {
  ss::grid_dependency_enter();
  build<true>(A);
}

struct Layout {
  size_t status, key[2], ints, total;
};
constexpr int kMaxBlocks = 1024;

static Layout layout(int n) {
  Layout L;
  size_t off = 0;
  L.status = off; off = align_up(off + kCleared);             // status, barrier, flags
  for (int i = 0; i < 2; ++i) { L.key[i] = off; off = align_up(off + static_cast<size_t>(n) * sizeof(uint64_t)); }
  L.ints = off; off = align_up(off + (static_cast<size_t>(11) * (n + 1) + kMaxBlocks) * 4);
  L.total = off;
  return L;
}

// One cluster of `blocks` (1 or 8), or a cooperative grid.
static int32_t launch(const Args& A, int blocks, bool cluster, cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(static_cast<unsigned>(blocks));
  cfg.blockDim = dim3(kThreads);
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  int n_attr = 0;
  if (cluster) {
    attr[n_attr].id = cudaLaunchAttributeClusterDimension;
    attr[n_attr].val.clusterDim.x = static_cast<unsigned>(blocks);
    attr[n_attr].val.clusterDim.y = attr[n_attr].val.clusterDim.z = 1;
    ++n_attr;
    if (pdl_enabled()) {
      attr[n_attr].id = cudaLaunchAttributeProgrammaticStreamSerialization;
      attr[n_attr].val.programmaticStreamSerializationAllowed = 1;
      ++n_attr;
    }
  } else {
    attr[n_attr].id = cudaLaunchAttributeCooperative;
    attr[n_attr].val.cooperative = 1;
    ++n_attr;
  }
  cfg.attrs = attr;
  cfg.numAttrs = static_cast<unsigned>(n_attr);
  const cudaError_t rc = cluster ? cudaLaunchKernelEx(&cfg, prefix_tree_cluster_kernel, A)
                                 : cudaLaunchKernelEx(&cfg, prefix_tree_grid_kernel, A);
  g_launch_count.fetch_add(1, std::memory_order_relaxed);
  if (rc != cudaSuccess || cudaPeekAtLastError() != cudaSuccess) {
    (void)cudaGetLastError();
    return SS_ERR_CUDA;
  }
  return SS_OK;
}

}  // namespace ptree
}  // namespace ss

extern "C" int32_t ss_prefix_tree_workspace_bytes(int32_t n_paths, int64_t total_tok, int32_t page_size,
                                                  size_t* out_bytes) {
  if (n_paths < 0 || n_paths > SS_PREFIX_TREE_MAX_PATHS || total_tok < 0 || page_size < 1 || !out_bytes)
    return SS_ERR_INVALID_ARG;
  *out_bytes = ss::ptree::layout(n_paths).total;
  return SS_OK;
}

extern "C" int32_t ss_build_prefix_tree(const int32_t* tok_ids, const int64_t* tok_offsets, int32_t n_paths,
                                        int64_t total_tok, int32_t page_size, int32_t* order_out,
                                        int32_t* path_leaf_node_out, int32_t* node_parent_out, int32_t* node_kv_len_out,
                                        int32_t* node_src_path_out, int32_t* node_src_offset_out,
                                        int32_t* num_nodes_out, void* workspace, size_t workspace_bytes, void* stream) {
  using namespace ss;
  using namespace ss::ptree;
  if (n_paths < 0 || n_paths > SS_PREFIX_TREE_MAX_PATHS || total_tok < 0 || page_size < 1) return SS_ERR_INVALID_ARG;
  if (!num_nodes_out || !workspace || reinterpret_cast<uintptr_t>(workspace) % kAlign) return SS_ERR_INVALID_ARG;
  const Layout L = layout(n_paths);
  if (workspace_bytes < L.total) return SS_ERR_WORKSPACE_TOO_SMALL;
  cudaStream_t st = as_stream(stream);
  char* ws = static_cast<char*>(workspace);
  // One block while it has a warp per position (its barrier is the cheapest).  A cluster of 8 blocks up to two positions per
  // warp and 16 MB of ids, which its 8 SMs read in 20 us: what the grid's barriers (1.5 us against 0.3, a dozen of them)
  // cost more.
  const int cluster = n_paths == 0 ? 0 : n_paths <= kWarps ? 1 : n_paths <= 512 && total_tok <= (1 << 22) ? 8 : 0;
  if ((cluster == 0 && cudaMemsetAsync(ws + L.status, 0, kCleared, st) != cudaSuccess) ||
      (n_paths == 0 && cudaMemsetAsync(num_nodes_out, 0, sizeof(int32_t), st) != cudaSuccess)) {
    (void)cudaGetLastError();
    return SS_ERR_CUDA;
  }
  if (n_paths == 0) return SS_OK;
  if (!tok_offsets || !order_out || !path_leaf_node_out || !node_parent_out || !node_kv_len_out || !node_src_path_out ||
      !node_src_offset_out || (total_tok > 0 && !tok_ids))
    return SS_ERR_INVALID_ARG;
  const int n = n_paths;
  Args A{};
  A.tok_ids = tok_ids;
  A.tok_offsets = tok_offsets;
  A.n = n;
  A.page = page_size;
  A.n_tiles = (n + kTile - 1) / kTile;
  A.status = reinterpret_cast<int32_t*>(ws + L.status);
  A.arrived = reinterpret_cast<unsigned int*>(ws + L.status + 64);
  A.flags = reinterpret_cast<unsigned int*>(ws + L.status + 128);
  for (int i = 0; i < 2; ++i) A.key[i] = reinterpret_cast<uint64_t*>(ws + L.key[i]);
  int* ints = reinterpret_cast<int*>(ws + L.ints);
  int** at[11] = {&A.perm[0], &A.perm[1], &A.gs, &A.ge, &A.lcp, &A.bmin, &A.c_start, &A.c_end, &A.outer, &A.cnt, &A.block_sum};
  for (int i = 0; i < 11; ++i) *at[i] = ints + static_cast<size_t>(i) * (n + 1);
  A.order = order_out;
  A.path_leaf_node = path_leaf_node_out;
  A.node_parent = node_parent_out;
  A.node_kv_len = node_kv_len_out;
  A.node_src_path = node_src_path_out;
  A.node_src_offset = node_src_offset_out;
  A.num_nodes = num_nodes_out;

  if (cluster > 0) return launch(A, cluster, true, st);
  int sms = sm_count_of_current_device();
  if (sms > kMaxBlocks) sms = kMaxBlocks;
  const int wanted = (n + kWarps - 1) / kWarps;
  return launch(A, wanted < sms ? wanted : sms, false, st);
}
