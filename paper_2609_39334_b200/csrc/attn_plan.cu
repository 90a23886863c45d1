// Device-side planner of ss_tree_attention: turns the tree + per-path arrays into work lists (tile items, leaf
// items), partial-slot assignments and per-path classes.  Running it on the device means the live path count can
// come straight from ss_dedup_paths without a host round trip.  Phases:
//   inputs  read and checked
//   nodes   keys before every node, depth check
//   paths   class of every path, membership counts of its chain nodes
//   tiles   per-node tile counts, KV splits, partial slots
//   scan    every prefix sum: decode ranks, tile items, partial slots, leaf items; capacity checks; totals
//   emit    the item lists and the per-decode-token arrays, a warp per path and per node
// Two forms of the same code:
//   small   (up to kSmallPlan nodes and paths)  one launch of a few blocks, each of which makes the WHOLE plan in its own shared
//           memory (redundantly: that needs no communication, and the phases cost their latency and instruction fetches whatever
//           the number of blocks) and then writes its share of the item lists
//   large   (any size)  one cluster makes the plan, its arrays in the workspace (2048 nodes and paths are what shared
//           memory holds), the cluster's hardware barrier between the phases; a second kernel writes the items, which
//           needs more warps than a cluster has
// Bound: the latency of the phases behind barriers, and of code that runs once (instruction fetches).  Measured, small: 922
// unique paths 20.9 -> 11.5 us, 256 verification paths 29.1 -> 8.2, 8 paths 12.0 -> 8.1 (against one block that shared the
// phases of a chain of five kernels and searched a path for every item).  Large, against that chain with its scan in one
// block, between events: 2912 paths 42.6 -> 29.2 us, 6400 57.8 -> 29.3, 25600 183 -> 54, 64000 452 -> 99; as ONE cooperative
// kernel with a barrier over the grid 40.7 and 43.9 for the first two (seven barriers, a memset, no overlap with its
// neighbours' launches).
// The header (status word first) is cleared and written by the planner itself.
#include <cooperative_groups.h>
#include "attn_plan.cuh"

namespace ss {
namespace attn {

namespace cg = cooperative_groups;

constexpr int kThreads = 1024;
constexpr int kSmallPlan = 2048;               // nodes and paths: two of each per thread
constexpr int kScanChunk = 2 * kThreads;       // entries of one block scan
constexpr int kLeafClasses = 24;               // of the last chunk of a leaf: 0 none; by length 1 .. 16 an only one, 17 .. 23 another
constexpr int kSums = 7;
constexpr int kLargeBlocks = 8;                // one cluster
constexpr int kEmitThreads = 256;

__device__ __forceinline__ int leaf_chunks(int len, int log2) { return (len + (1 << log2) - 1) >> log2; }

__device__ __forceinline__ int live_paths(const Params& P) {
  int live = P.num_paths;
  if (P.num_paths_dev) {
    live = *P.num_paths_dev;
    if (live < 0) live = 0;
    if (live > P.num_paths) live = P.num_paths;
  }
  return live;
}

// KV splits of a root, while there are fewer tile items (`total_tiles`) than it takes to keep the device busy.
__device__ __forceinline__ void node_split(const Params& P, int len, int total_tiles, int& splits, int& split_len) {
  if (total_tiles >= P.target_tiles) return;
  int want = ceil_div(P.target_tiles, total_tiles);
  const int most = min(len / kMinSplitLen, kMaxRootSplits);
  if (want > most) want = most;
  if (want > 1) {
    split_len = ceil_div(ceil_div(len, want), kKvTile) * kKvTile;
    splits = ceil_div(len, split_len);
  }
}

// Seven exclusive scans at once over the block's entries 2 tid, 2 tid + 1 (v -> positions), and the totals; with RANK, in the
// same two barriers, the rank of each entry among all of them, larger classes cls[] first (order[]: deterministic, but not
// index order within a class).
static_assert(8 + kLeafClasses <= 32, "a warp for each class, behind the first 8");
struct BlockScan {
  int tot[kSums][32];          // per warp, then exclusive over the warps
  int total[kSums];
  int hist[kLeafClasses][64];  // per class and group of 32 entries, then exclusive over the groups
  int cls_total[kLeafClasses];
};
template <bool RANK>
__device__ __forceinline__ void block_scan(BlockScan& S, int (&v)[kSums][2], const int (&cls)[2], int (&order)[2]) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  int sum[kSums], x[kSums];
#pragma unroll
  for (int k = 0; k < kSums; ++k) x[k] = sum[k] = v[k][0] + v[k][1];
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
#pragma unroll
    for (int k = 0; k < kSums; ++k) {
      const int y = __shfl_up_sync(0xffffffffu, x[k], o);
      if (lane >= o) x[k] += y;
    }
  }
  if (lane == 31) {
#pragma unroll
    for (int k = 0; k < kSums; ++k) S.tot[k][warp] = x[k];
  }
  int in_group[2] = {0, 0};
  if (RANK) {
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const uint32_t peers = __match_any_sync(0xffffffffu, cls[e]);
      in_group[e] = __popc(peers & ((1u << lane) - 1u));
      if (in_group[e] == 0) S.hist[cls[e]][2 * warp + e] = __popc(peers);   // (the rest was cleared by the caller)
    }
  }
  __syncthreads();
  if (warp < kSums) {
    const int t = S.tot[warp][lane];
    int y = t;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int z = __shfl_up_sync(0xffffffffu, y, o);
      if (lane >= o) y += z;
    }
    S.tot[warp][lane] = y - t;
    if (lane == 31) S.total[warp] = y;
  } else if (RANK && warp >= 8 && warp < 8 + kLeafClasses) {
    int* h = S.hist[warp - 8];
    const int a = h[2 * lane], b = h[2 * lane + 1];
    int y = a + b;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int z = __shfl_up_sync(0xffffffffu, y, o);
      if (lane >= o) y += z;
    }
    h[2 * lane] = y - a - b;
    h[2 * lane + 1] = y - b;
    if (lane == 31) S.cls_total[warp - 8] = y;
  }
  __syncthreads();
#pragma unroll
  for (int k = 0; k < kSums; ++k) {
    const int first = S.tot[k][warp] + x[k] - sum[k];
    v[k][1] = first + v[k][0];
    v[k][0] = first;
  }
  if (RANK) {
    int above = lane < kLeafClasses ? S.cls_total[lane] : 0;    // lane r: entries of the classes > r
    const int own = above;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int z = __shfl_down_sync(0xffffffffu, above, o);
      if (lane + o < 32) above += z;
    }
    above -= own;
#pragma unroll
    for (int e = 0; e < 2; ++e) order[e] = __shfl_sync(0xffffffffu, above, cls[e]) + S.hist[cls[e]][2 * warp + e] + in_group[e];
  }
}

// The plan up to the item lists.  `A`: its arrays, in shared memory (small) or in the workspace; `bad_phase`: a word per phase
// in the block's shared memory; `totals` (tiles of the shared nodes, rows of GENERIC paths, shorter items of the private leaves of
// a kv head): in shared memory, of block 0 of the cluster in the large form.  All start at zero.  False: it failed, the status says why.
template <bool LARGE>
__device__ __forceinline__ bool make_plan(const Params& P, const PlanArrays& A, PlanHeader* hdr, BlockScan& S, int* bad_phase,
                                          int* totals) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int N = P.num_nodes, NP = P.num_paths, Hkv = P.Hkv, tpt = P.tok_per_tile;
  const int first = LARGE ? static_cast<int>(blockIdx.x) * kThreads + tid : tid;
  const int stride = LARGE ? kLargeBlocks * kThreads : kThreads;
  int phase = 0;
  // Ends a phase: true in every thread of every block that plans if `bad` was set in any of them.  (The large form tells
  // every block, in a word of the phase's own: a block that is already in the next phase must not change what others read.)
  auto phase_failed = [&](bool bad, int code) -> bool {
    if (LARGE) {
      if (bad) {
        for (int r = 0; r < kLargeBlocks; ++r) *cg::this_cluster().map_shared_rank(&bad_phase[phase], r) = 1;
        set_status(&hdr->status, code);
      }
      cg::this_cluster().sync();
      return bad_phase[phase++] != 0;
    }
    const bool any = __syncthreads_or(bad) != 0;
    if (any && tid == 0) hdr->status = code;
    return any;
  };

  // ---- inputs (the per-path arrays up to their capacity, beside the live count: one trip) ---------------------------------
  const int live = live_paths(P);
  bool bad = false;
#pragma unroll 1
  for (int i = first; i < max(N, NP); i += stride) {           // (node i and path i: their loads go out together)
    const int n = min(i, N - 1), p = min(i, NP - 1);
    int parent = 0, len = 0, leaf = 0, T = 0;
    int64_t o0 = 0, o1 = 0, r0 = 0, r1 = 0, src = 0;
    if (N > 0) {
      parent = P.node_parent[n];
      len = P.node_kv_len[n];
      o0 = P.node_page_offsets[n];
      o1 = P.node_page_offsets[n + 1];
    }
    if (NP > 0) {
      leaf = P.path_leaf_node[p];
      T = P.path_q_len[p];
      r0 = P.q_offsets[p];
      r1 = P.q_offsets[p + 1];
      src = P.q_src_offsets ? P.q_src_offsets[p] : r0;
    }
    if (i < N) {
      bad = bad || parent >= n || parent < -1 || len < 0 || o1 < o0 || (o1 - o0) * kPage < len || o1 > P.total_node_pages || o0 < 0;
      if (!LARGE) {
        A.n_parent[n] = parent;
        A.n_len[n] = len;
        A.n_page0[n] = static_cast<int32_t>(o0);
      }
      A.n_first[n] = 0x7fffffff;
      A.n_last[n] = -1;
      A.n_paths[n] = A.n_dec[n] = 0;
    }
    if (i < NP) {
      bool ok = leaf >= 0 && leaf < N && T >= 1 && r1 - r0 == T && r0 >= 0 && r1 <= P.total_q;
      if (P.q_src_offsets) ok = ok && src >= 0 && src + T <= P.q_src_rows && src + T <= 0x7fffffffLL;
      bad = bad || (i < live && !ok);
      if (!LARGE) {
        A.p_leaf[p] = leaf;
        A.p_T[p] = T;
        A.p_row[p] = static_cast<int32_t>(r0);
        A.p_src[p] = static_cast<int32_t>(src);
      }
    }
  }
  if (P.flags & SS_FLAG_VALIDATE) {
    for (int64_t i = first; i < P.total_node_pages; i += stride) {
      const int pg = P.node_pages[i];
      bad = bad || pg < 0 || pg >= P.num_pages;
    }
  }
  if (phase_failed(bad, SS_ERR_BAD_INPUT)) return false;

  // ---- nodes: keys before the node (parents come first, so every walk ends) ---------------------------------------------------
  bad = false;
#pragma unroll 1
  for (int n = first; n < N; n += stride) {
    int d = 1, start = 0;
#pragma unroll 1
    for (int a = A.n_parent[n]; a >= 0 && d <= SS_MAX_DEPTH; a = A.n_parent[a]) { start += A.n_len[a]; ++d; }
    bad = bad || d > SS_MAX_DEPTH;
    A.n_start[n] = start;
  }
  if (phase_failed(bad, SS_ERR_UNSUPPORTED)) return false;

  // ---- paths: class, membership of every chain node (lanes with the same node are counted together) -----------------------
#pragma unroll 1
  for (int p0 = first - tid; p0 < live; p0 += stride) {
    const int p = p0 + tid;
    const int leaf = p < live ? A.p_leaf[p] : -1, T = p < live ? A.p_T[p] : 0;
    const bool force = (P.flags & SS_FLAG_FORCE_GENERIC) != 0;
    const bool dec = leaf >= 0 && T == 1 && P.G <= 16 && !force;
    const uint32_t decs = __ballot_sync(0xffffffffu, dec);
    bool whole = true;                                         // inner nodes are whole pages
    int a = leaf;
#pragma unroll 1
    while (__any_sync(0xffffffffu, a >= 0)) {
      const uint32_t peers = __match_any_sync(0xffffffffu, a);
      if (a >= 0) {
        if ((peers & ((1u << lane) - 1u)) == 0) {
          atomicMin(&A.n_first[a], p);
          atomicMax(&A.n_last[a], p + 31 - __clz(peers) - lane);
          atomicAdd(&A.n_paths[a], __popc(peers));
          if (peers & decs) atomicAdd(&A.n_dec[a], __popc(peers & decs));
        }
        if (a != leaf && A.n_len[a] % kPage) whole = false;
        a = A.n_parent[a];
      }
    }
    if (leaf >= 0) {
      const int cls = dec ? kClassDecode : (force || T == 1 || !whole ? kClassGeneric : kClassChain);
      A.p_class[p] = cls;
      if (cls == kClassGeneric) atomicAdd(&totals[1], T);
    }
  }
  phase_failed(false, SS_OK);

  // ---- nodes: tiles (what other blocks' atomics counted is read from L2) ----------------------------------------------------
  auto count = [](const int32_t* c) { return LARGE ? __ldcg(c) : *c; };
  bad = false;
  int mine = 0, my_leaves = 0;
#pragma unroll 1
  for (int n = first; n < N; n += stride) {
    const int np = count(A.n_paths + n), nd = count(A.n_dec + n), p0 = count(A.n_first + n);
    bad = bad || (np > 0 && count(A.n_last + n) - p0 + 1 != np);
    int tiles = 0;
    if (nd > 0 && A.n_len[n] > 0) {
      if (np == 1 && A.p_leaf[p0] == n)
        my_leaves += leaf_chunks(A.n_len[n], kLeafChunkLog2);
      else
        tiles = ceil_div(nd, tpt);
    }
    A.n_tiles[n] = tiles;
    mine += tiles;
  }
  mine = static_cast<int>(__reduce_add_sync(0xffffffffu, static_cast<unsigned>(mine)));
  if (lane == 0 && mine) atomicAdd(&totals[0], mine);
  my_leaves = static_cast<int>(__reduce_add_sync(0xffffffffu, static_cast<unsigned>(my_leaves)));
  if (lane == 0 && my_leaves) atomicAdd(&totals[2], my_leaves);
  if (phase_failed(bad, SS_ERR_BAD_INPUT)) return false;

  // ---- nodes: KV splits, partial slots ------------------------------------------------------------------------------------------
  const int total_tiles = totals[0] * Hkv;
  const int leaf_log2 = static_cast<int64_t>(totals[2]) * Hkv >= P.leaf_warps ? kLeafChunkLog2Many : kLeafChunkLog2;
#pragma unroll 1
  for (int n = first; n < N; n += stride) {
    const int len = A.n_len[n], tiles = A.n_tiles[n];
    int splits = 1, own = 0, split_len = len;
    if (tiles > 0) {
      if (A.n_parent[n] < 0) node_split(P, len, total_tiles, splits, split_len);
      own = splits;
    } else if (count(A.n_dec + n) > 0 && len > 0) {
      own = leaf_chunks(len, leaf_log2);                       // private leaf of one decode path
    }
    A.n_splits[n] = splits;
    A.n_split_len[n] = split_len;
    A.n_own[n] = own;
  }
  phase_failed(false, SS_OK);

  // ---- every prefix sum: entries 2 tid, 2 tid + 1 of the nodes and of the paths, a chunk per block at a time ----------------
  // sums: items of the roots, of the other nodes, decode paths, partial slots, whole leaf chunks, chain items, last chunks
  const int n_chunks = LARGE ? max(1, ceil_div(max(N, live), kScanChunk)) : 1;
#pragma unroll 1
  for (int chunk = LARGE ? blockIdx.x : 0; chunk < n_chunks; chunk += LARGE ? gridDim.x : 1) {
    int v[kSums][2], cls[2] = {0, 0}, order[2];
#pragma unroll 1
    for (int e = 0; e < 2; ++e) {
      const int i = chunk * kScanChunk + 2 * tid + e;
      int root_items = 0, node_items = 0, slots = 0, full = 0, chain = 0, dec = 0, c = 0;
      if (i < N) {
        int off = 0;
#pragma unroll 1
        for (int a = A.n_parent[i]; a >= 0; a = A.n_parent[a]) off += A.n_own[a];
        A.n_level[i] = off;
        const int items = A.n_tiles[i] * A.n_splits[i] * Hkv;
        if (A.n_parent[i] < 0) root_items = items; else node_items = items;
      }
      if (i < live) {
        const int leaf = A.p_leaf[i], len = A.n_len[leaf];
        if (A.p_class[i] == kClassDecode) {
          dec = 1;
#pragma unroll 1
          for (int a = leaf; a >= 0; a = A.n_parent[a]) slots += A.n_own[a];
          if (count(A.n_paths + leaf) == 1 && len > 0) {
            full = len >> leaf_log2;
            c = ceil_div(len - (full << leaf_log2), kPage);
            // leaves of several chunks before those of one, whose end is cheaper: the merge of several, fence and all, is not
            // to be what the kernel ends with (922 leaves of 32 to 512 keys in chunks of 256, the step: 92.5 -> 88.5 us)
            if (!LARGE && c > 0) c = full > 0 ? 16 + (c + 4) / 5 : (c + 1) / 2;
            if (!LARGE && P.short_first && c > 0) c = kLeafClasses - c;
          }
        } else if (A.p_class[i] == kClassChain) {
          chain = ceil_div(A.p_T[i], tpt) * Hkv;
        }
      }
      const int last = c > 0 ? 1 : 0;
      if (e == 0) {
        v[0][0] = root_items; v[1][0] = node_items; v[2][0] = dec; v[3][0] = slots; v[4][0] = full; v[5][0] = chain; v[6][0] = last; cls[0] = c;
      } else {
        v[0][1] = root_items; v[1][1] = node_items; v[2][1] = dec; v[3][1] = slots; v[4][1] = full; v[5][1] = chain; v[6][1] = last; cls[1] = c;
      }
    }
    block_scan<!LARGE>(S, v, cls, order);
    const int roots = LARGE ? 0 : S.total[0];
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const int i = chunk * kScanChunk + 2 * tid + e;
      if (i < N) A.n_base[i] = A.n_parent[i] < 0 ? v[0][e] : roots + v[1][e];   // the roots' items come first
      if (i < live) {
        A.p_rank[i] = v[2][e];
        A.p_slot[i] = v[3][e];
        A.p_items[i] = A.p_class[i] == kClassChain ? v[5][e] : v[4][e] + (LARGE ? v[6][e] : 0);
        if (!LARGE) A.p_last[i] = cls[e] > 0 ? order[e] : -1;
      }
    }
    if (LARGE && tid < kSums) A.sums[chunk * 8 + tid] = S.total[tid];
    __syncthreads();
  }
  if (LARGE) {
    phase_failed(false, SS_OK);
    // totals, and for each chunk of this block what lies in front of it
#pragma unroll 1
    for (int chunk = blockIdx.x; chunk == static_cast<int>(blockIdx.x) || chunk < n_chunks; chunk += gridDim.x) {
      if (warp < kSums) {
        int before = 0, all = 0;
        for (int c = lane; c < n_chunks; c += 32) {
          const int x = __ldcg(A.sums + c * 8 + warp);
          all += x;
          if (c < chunk) before += x;
        }
        before = static_cast<int>(__reduce_add_sync(0xffffffffu, static_cast<unsigned>(before)));
        all = static_cast<int>(__reduce_add_sync(0xffffffffu, static_cast<unsigned>(all)));
        if (lane == 0) {
          S.tot[warp][0] = before;
          S.total[warp] = all;
        }
      }
      __syncthreads();
      if (chunk < n_chunks) {
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const int i = chunk * kScanChunk + 2 * tid + e;
          if (i < N) A.n_base[i] += A.n_parent[i] < 0 ? S.tot[0][0] : S.total[0] + S.tot[1][0];
          if (i < live) {
            A.p_rank[i] += S.tot[2][0];
            A.p_slot[i] += S.tot[3][0];
            A.p_items[i] += A.p_class[i] == kClassChain ? S.tot[5][0] : S.tot[4][0] + S.tot[6][0];
          }
        }
      }
      __syncthreads();
    }
  }
  if (tid == 0 && (!LARGE || blockIdx.x == 0)) {
    const int* total = S.total;
    const int n_stacked = total[0] + total[1], n_full = total[4] * Hkv, n_leaf_items = n_full + total[6] * Hkv;
    const bool small_ws = total[2] > P.caps.dec || total[3] > P.caps.slots || n_leaf_items > P.caps.leaf_items ||
                          n_stacked + total[5] > P.caps.tile_items;
    if (small_ws) hdr->status = SS_ERR_WORKSPACE_TOO_SMALL;    // nothing is emitted, the executors see the status and do nothing
    hdr->live_paths = live;
    hdr->n_dec = total[2];
    hdr->n_slots = total[3];
    hdr->n_stacked_items = n_stacked;
    hdr->n_generic_rows = totals[1];
    hdr->n_full_leaf_items = n_full;
    hdr->leaf_log2 = leaf_log2;
    hdr->n_leaf_items = small_ws ? 0 : n_leaf_items;
    hdr->n_tile_items = small_ws ? 0 : n_stacked + total[5];
  }
  return true;
}

// The item lists and the per-decode-token arrays: a warp per path and per node, of all blocks of the grid.
template <bool LARGE>
__device__ __forceinline__ void emit_items(const Params& P, const PlanArrays& A, const PlanHeader* hdr) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int N = P.num_nodes, Hkv = P.Hkv, tpt = P.tok_per_tile;
  const int live = hdr->live_paths, n_stacked = hdr->n_stacked_items, n_full = hdr->n_full_leaf_items, leaf_log2 = hdr->leaf_log2;
  const int full0 = !LARGE && P.short_first ? hdr->n_leaf_items - n_full : 0, last0 = P.short_first ? 0 : n_full;
  const int wid = blockIdx.x * (blockDim.x / 32) + warp, nw = gridDim.x * (blockDim.x / 32);
  auto page0_of = [&](int n) { return LARGE ? static_cast<int32_t>(P.node_page_offsets[n]) : A.n_page0[n]; };
  if (wid == 0 && lane == 0) P.dec_slot_base[hdr->n_dec] = hdr->n_slots;
#pragma unroll 1
  for (int p = wid; p < live; p += nw) {
    const int leaf = A.p_leaf[p], len = A.n_len[leaf], cls = A.p_class[p], L = A.n_start[leaf] + len;
    if (lane == 0) {                                           // (read by the generic rows and the exact second pass)
      if (!LARGE) P.path_class[p] = cls;
      P.path_kv_len[p] = L;
    }
    const int row = LARGE ? static_cast<int32_t>(P.q_offsets[p]) : A.p_row[p];
    const int src = !LARGE ? A.p_src[p] : P.q_src_offsets ? static_cast<int32_t>(P.q_src_offsets[p]) : row;
    if (cls == kClassDecode) {
      const int rank = A.p_rank[p], slot = A.p_slot[p];
      const bool own_leaf = A.n_paths[leaf] == 1 && len > 0;
      if (lane == 0) {
        P.dec_tok[rank] = row;
        P.dec_src[rank] = src;
        P.dec_slot_base[rank] = slot;
        P.dec_leaf_chunks[rank] = own_leaf ? leaf_chunks(len, leaf_log2) : 0;
      }
      for (int g = lane; g < Hkv; g += 32) P.leaf_arrive[static_cast<int64_t>(rank) * Hkv + g] = 0;
      if (!own_leaf) continue;
      // The leaf kernel hands its items out in this order.  Small form: whole chunks first, then the last chunks of all leaves,
      // longest first, so that the short ones level out the warps' ends (922 leaves of 32 to 512 keys: 71.6 -> 68.9 us).  Large
      // form: leaf after leaf; with many items per warp the order by length only costs (6550 leaves of 128 to 1024 keys: 2.46 ms,
      // whole chunks first 2.43, leaf after leaf 2.37).  Where the rows go over the bus as the leaves are done, the small form
      // turns its order round, so that the bus is not idle until the longest ones are (a step of 1024 paths from host buffers
      // 227 -> 214 us)
      const int page0 = page0_of(leaf), full = len >> leaf_log2, n_items = leaf_chunks(len, leaf_log2) * Hkv;
      const int last = LARGE ? 0 : A.p_last[p];
#pragma unroll 1
      for (int x = lane; x < n_items; x += 32) {
        const int c = x / Hkv, g = x - c * Hkv;
        LeafItem it;
        it.page0 = page0 + ((c << leaf_log2) / kPage);
        it.node = leaf;
        it.g = g;
        it.kv_begin = c << leaf_log2;
        it.kv_end = min(len, (c + 1) << leaf_log2);
        it.slot = slot + A.n_level[leaf] + c;
        it.q_src = src;
        it.dec = rank;
        P.leaf_items[LARGE || c < full ? full0 + A.p_items[p] * Hkv + x : last0 + last * Hkv + g] = it;
      }
    } else if (cls == kClassChain) {
      const int T = A.p_T[p], tiles = ceil_div(T, tpt);
#pragma unroll 1
      for (int x = lane; x < tiles * Hkv; x += 32) {
        const int g = x / tiles, t = x - g * tiles;
        TileItem it;
        it.node = leaf;
        it.tok0 = row + t * tpt;
        it.n_tok = min(tpt, T - t * tpt);
        it.kind_g = (kItemChain << 16) | g;
        it.kv_begin = 0;
        it.limit0 = L - T + t * tpt + 1;
        it.kv_end = max(0, min(L, it.limit0 + it.n_tok - 1));
        it.slot_off = -1;
        it.src0 = src + t * tpt;
        it.pad = 0;
        P.tile_items[n_stacked + A.p_items[p] + x] = it;
      }
    }
  }
#pragma unroll 1
  for (int n = wid; n < N; n += nw) {
    if (!LARGE && lane == 0) P.node_start[n] = A.n_start[n];
    const int tiles = A.n_tiles[n];
    if (tiles == 0) continue;
    const int page0 = page0_of(n), splits = A.n_splits[n], split_len = A.n_split_len[n], len = A.n_len[n], nd = A.n_dec[n],
              rank0 = A.p_rank[A.n_first[n]];
#pragma unroll 1
    for (int x = lane; x < tiles * splits * Hkv; x += 32) {
      const int rest = x / splits, split = x - rest * splits, tile = rest / Hkv, g = rest - tile * Hkv;
      TileItem it;
      it.node = n;
      it.tok0 = rank0 + tile * tpt;
      it.n_tok = min(tpt, nd - tile * tpt);
      it.kind_g = (kItemStacked << 16) | g;
      it.kv_begin = split * split_len;
      it.kv_end = min(len, (split + 1) * split_len);
      it.limit0 = it.kv_end;
      it.slot_off = A.n_level[n] + split;
      it.src0 = page0;
      it.pad = 0;
      P.tile_items[A.n_base[n] + x] = it;
    }
  }
}

__global__ void __launch_bounds__(kThreads) plan_small_kernel(const __grid_constant__ Params P) {
  ss::grid_dependency_enter();
  extern __shared__ __align__(16) int32_t plan_smem[];
  __shared__ PlanHeader s_hdr;
  __shared__ BlockScan s_scan;
  __shared__ int s_totals[3];
  const int tid = threadIdx.x;
  PlanArrays A;
  int32_t* w = plan_smem;
  for (int x = 0; x < kPlanNodeArrays + kPlanNodeInputs; ++x, w += P.num_nodes) A.node_array(x) = w;
  for (int x = 0; x < kPlanPathArrays + kPlanPathInputs; ++x, w += P.num_paths) A.path_array(x) = w;
  A.sums = nullptr;
  for (int x = tid; x < kPlanHeaderWords; x += kThreads) reinterpret_cast<int32_t*>(&s_hdr)[x] = 0;
  for (int x = tid; x < kLeafClasses * 64; x += kThreads) (&s_scan.hist[0][0])[x] = 0;
  if (tid < 3) s_totals[tid] = 0;
  SS_STAMP_BEGIN(P.hdr, 0);
  make_plan<false>(P, A, &s_hdr, s_scan, nullptr, s_totals);
  __syncthreads();
  if (s_hdr.status == SS_OK) emit_items<false>(P, A, &s_hdr);
  if (blockIdx.x != 0) return;
#ifdef SS_STAMPS
  __syncthreads();
  if (tid == 0) { s_hdr.stamp[0] = P.hdr->stamp[0]; s_hdr.stamp[1] = ss_globaltimer(); }
#endif
  __syncthreads();
  for (int x = tid; x < kPlanHeaderWords; x += kThreads)
    reinterpret_cast<int32_t*>(P.hdr)[x] = reinterpret_cast<const int32_t*>(&s_hdr)[x];
}

__global__ void __cluster_dims__(kLargeBlocks, 1, 1) __launch_bounds__(kThreads) plan_large_kernel(const __grid_constant__ Params P) {
  ss::grid_dependency_enter();
  __shared__ BlockScan s_scan;
  __shared__ int s_bad[8], s_totals[3];
  const int tid = threadIdx.x;
  if (tid < 8) s_bad[tid] = 0;
  if (tid < 3) s_totals[tid] = 0;
  if (blockIdx.x == 0 && tid < kPlanHeaderWords) reinterpret_cast<int32_t*>(P.hdr)[tid] = 0;
  cg::this_cluster().sync();
  SS_STAMP_BEGIN(P.hdr, 0);
  make_plan<true>(P, P.plan, P.hdr, s_scan, s_bad, cg::this_cluster().map_shared_rank(s_totals, 0));
}

__global__ void __launch_bounds__(kEmitThreads) plan_emit_kernel(const __grid_constant__ Params P) {
  ss::grid_dependency_enter();
  if (P.hdr->status == SS_OK) emit_items<true>(P, P.plan, P.hdr);
  SS_STAMP_END(P.hdr, 1);
}

int32_t launch_plan(const Params& P, cudaStream_t st) {
  const int N = P.num_nodes, NP = P.num_paths;
  if (N <= kSmallPlan && NP <= kSmallPlan) {                   // (this kernel writes the whole header itself)
    auto smem = [](int n, int np) { return static_cast<size_t>(4) * (static_cast<size_t>(n) * (kPlanNodeArrays + kPlanNodeInputs) +
                                         static_cast<size_t>(np) * (kPlanPathArrays + kPlanPathInputs)) + 64; };
    static bool configured[kDeviceSlots] = {false};
    const int dev_slot = current_device_slot();
    if (dev_slot < 0 || !configured[dev_slot]) {
      if (cudaFuncSetAttribute(plan_small_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               static_cast<int>(smem(kSmallPlan, kSmallPlan))) != cudaSuccess) {
        (void)cudaGetLastError();
        return SS_ERR_CUDA;
      }
      if (dev_slot >= 0) configured[dev_slot] = true;
    }
    int blocks = (N + NP + 31) / 32;                           // what is left to share is the emission, a warp per path and node
    blocks = blocks < 1 ? 1 : (blocks > 64 ? 64 : blocks);
    SS_LAUNCH(plan_small_kernel, blocks, kThreads, smem(N, NP), st, P);
    return SS_OK;
  }
  SS_LAUNCH(plan_large_kernel, kLargeBlocks, kThreads, 0, st, P);
  int64_t blocks = (static_cast<int64_t>(N) + NP + kEmitThreads / 32 - 1) / (kEmitThreads / 32);
  if (blocks > P.sms * 8) blocks = P.sms * 8;
  SS_LAUNCH(plan_emit_kernel, static_cast<int>(blocks), kEmitThreads, 0, st, P);
  return SS_OK;
}

}  // namespace attn
}  // namespace ss
