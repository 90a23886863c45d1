// Device-side planner of ss_tree_attention: turns the tree + per-path arrays into work lists (tile items, leaf
// items), partial-slot assignments and per-path classes.  Running it on the device means the live path count can
// come straight from ss_dedup_paths without a host round trip.  Four phases:
//   nodes   depth and prefix length of every node, range checks, counters reset
//   paths   class and key length of every path, membership counts of its chain nodes
//   scan    (one block) every prefix sum: decode ranks, per-node tile items and KV splits, partial slots, leaf
//           items, chain items; capacity checks; totals into the header
//   emit    writes the item lists and the per-decode-token arrays
// Trees of up to kSmallPlan nodes and paths are planned in ONE launch of a few blocks, each of which makes the WHOLE plan in
// its own shared memory (redundantly: that needs no communication, and the phases cost their latency and instruction
// fetches whatever the number of blocks) and then writes its share of the item lists.  Larger inputs take four launches
// (nodes, paths and emit grid-parallel, scan in one block).  Bound: the latency of seven phases behind barriers, and of
// code that runs once (instruction fetches).  Measured, against one block that shared the phases of the general path and
// searched a path for every item: 922 unique paths 20.9 -> 11.5 us, 256 verification paths 29.1 -> 8.2, 8 paths 12.0 -> 8.1.
// The header (status word first) is cleared by the host-side launcher before the first of the four kernels; the
// small planner builds it in shared memory and its block 0 writes it out whole.
#include "attn_plan.cuh"

namespace ss {
namespace attn {

constexpr int kScanThreads = 1024;
constexpr int kGridThreads = 256;

// In-place exclusive scan of a[0..n) by one whole block: every thread sums a contiguous chunk, the chunk sums are
// scanned across the block, then every thread rewrites its chunk.  Returns the total to every thread.
__device__ int block_excl_scan_chunks(int32_t* a, int n) {
  __shared__ int warp_tot[32];
  __shared__ int total_s;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int chunk = (n + blockDim.x - 1) / blockDim.x;
  const int lo = min(n, static_cast<int>(threadIdx.x) * chunk), hi = min(n, lo + chunk);
  __syncthreads();
  int sum = 0;
  for (int i = lo; i < hi; ++i) sum += a[i];
  int x = sum;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) warp_tot[warp] = x;
  __syncthreads();
  if (warp == 0) {
    int t = lane < nw ? warp_tot[lane] : 0;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, t, o);
      if (lane >= o) t += y;
    }
    warp_tot[lane] = t;
    if (lane == 31) total_s = t;
  }
  __syncthreads();
  int run = (warp ? warp_tot[warp - 1] : 0) + x - sum;
  for (int i = lo; i < hi; ++i) {
    const int v = a[i];
    a[i] = run;
    run += v;
  }
  __syncthreads();
  return total_s;
}

// Two scans of arrays in GLOBAL memory of up to 16 entries per thread at once: a thread keeps its 16 consecutive entries of
// each array in registers (128-bit loads, all issued before the first is used; 128-bit stores), so a pair of scans
// costs two trips to memory instead of the six of two staged scans.  The arrays must be 16-byte aligned.
constexpr int kScanRegs = 16;
__device__ void block_excl_scan2_regs(int32_t* a0, int32_t* a1, int n, int (&total)[2]) {   // (two arrays per call: 32 of a thread's 64 registers)
  __shared__ int warp_tot4[32][2];
  __shared__ int total4_s[2];
  int32_t* a[2] = {a0, a1};
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int lo = static_cast<int>(threadIdx.x) * kScanRegs;
  int v[2][kScanRegs];
  __syncthreads();
#pragma unroll
  for (int k = 0; k < 2; ++k) {
#pragma unroll
    for (int i = 0; i < kScanRegs; i += 4) {
      if (lo + i + 4 <= n) {
        const int4 q = *reinterpret_cast<const int4*>(a[k] + lo + i);
        v[k][i] = q.x; v[k][i + 1] = q.y; v[k][i + 2] = q.z; v[k][i + 3] = q.w;
      } else {
#pragma unroll
        for (int j = 0; j < 4; ++j) v[k][i + j] = (lo + i + j < n) ? a[k][lo + i + j] : 0;
      }
    }
  }
  int sum[2], x[2];
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    sum[k] = 0;
#pragma unroll
    for (int i = 0; i < kScanRegs; ++i) sum[k] += v[k][i];
    x[k] = sum[k];
  }
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const int y = __shfl_up_sync(0xffffffffu, x[k], o);
      if (lane >= o) x[k] += y;
    }
  }
  if (lane == 31) {
#pragma unroll
    for (int k = 0; k < 2; ++k) warp_tot4[warp][k] = x[k];
  }
  __syncthreads();
  if (warp == 0) {
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      int t = lane < nw ? warp_tot4[lane][k] : 0;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, t, o);
        if (lane >= o) t += y;
      }
      warp_tot4[lane][k] = t;
      if (lane == 31) total4_s[k] = t;
    }
  }
  __syncthreads();
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    int run = (warp ? warp_tot4[warp - 1][k] : 0) + x[k] - sum[k];
#pragma unroll
    for (int i = 0; i < kScanRegs; i += 4) {
      int4 q;
      q.x = run; run += v[k][i];
      q.y = run; run += v[k][i + 1];
      q.z = run; run += v[k][i + 2];
      q.w = run; run += v[k][i + 3];
      if (lo + i + 4 <= n) {
        *reinterpret_cast<int4*>(a[k] + lo + i) = q;
      } else {
        if (lo + i < n) a[k][lo + i] = q.x;
        if (lo + i + 1 < n) a[k][lo + i + 1] = q.y;
        if (lo + i + 2 < n) a[k][lo + i + 2] = q.z;
      }
    }
    total[k] = total4_s[k];
  }
  __syncthreads();
}

// The same scan for an array in GLOBAL memory: it goes through the block's staging buffer in shared memory when it
// fits (coalesced in, scanned on chip, coalesced out) - every thread walking its own contiguous chunk of a global
// array makes each load touch 32 different sectors, which cost the one-block scan kernel most of its time.
constexpr int kScanStage = 16384;                  // entries of the staging buffer (64 KB, dynamic shared memory)
__device__ int block_excl_scan(int32_t* a, int n, int32_t* stage) {
  if (n > kScanStage) return block_excl_scan_chunks(a, n);
  __syncthreads();
  for (int i = threadIdx.x; i < n; i += blockDim.x) stage[i] = a[i];
  const int total = block_excl_scan_chunks(stage, n);      // (starts and ends with a barrier)
  for (int i = threadIdx.x; i < n; i += blockDim.x) a[i] = stage[i];
  __syncthreads();
  return total;
}

// Block-uniform read of the status word (every thread gets the same answer, so an early return cannot leave
// part of the block waiting at a later barrier).
__device__ bool block_failed(const PlanHeader* hdr) {
  __shared__ int s_status;
  __syncthreads();
  if (threadIdx.x == 0) s_status = *reinterpret_cast<const volatile int32_t*>(&hdr->status);
  __syncthreads();
  return s_status != SS_OK;
}

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

// ---- nodes: depth and number of keys before the node -------------------------------------------------------------
__device__ __forceinline__ void plan_nodes_phase(const Params& P) {
  PlanHeader* hdr = P.hdr;
  const int64_t gtid = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  const int64_t gsize = static_cast<int64_t>(gridDim.x) * blockDim.x;
  if (gtid == 0) hdr->live_paths = live_paths(P);
  for (int64_t n64 = gtid; n64 < P.num_nodes; n64 += gsize) {
    const int n = static_cast<int>(n64);
    int d = 0, start = 0;
    int a = P.node_parent[n];
    bool bad = (a >= n || a < -1 || P.node_kv_len[n] < 0);
    while (!bad && a >= 0 && d < SS_MAX_DEPTH) {
      start += P.node_kv_len[a];
      ++d;
      const int na = P.node_parent[a];
      if (na >= a || na < -1) { bad = true; break; }
      a = na;
    }
    if (bad) set_status(&hdr->status, SS_ERR_BAD_INPUT);
    else if (a >= 0 || d + 1 > SS_MAX_DEPTH) set_status(&hdr->status, SS_ERR_UNSUPPORTED);
    const int64_t np = P.node_page_offsets[n + 1] - P.node_page_offsets[n];
    if (!bad && (np < 0 || np * kPage < P.node_kv_len[n] || P.node_page_offsets[n + 1] > P.total_node_pages ||
                 P.node_page_offsets[n] < 0))
      set_status(&hdr->status, SS_ERR_BAD_INPUT);
    P.node_depth[n] = d;
    P.node_start[n] = start;
    P.node_first[n] = 0x7fffffff;
    P.node_last[n] = -1;
    P.node_npaths[n] = 0;
    P.node_ndec[n] = 0;
  }
  if (P.flags & SS_FLAG_VALIDATE) {
    for (int64_t i = gtid; i < P.total_node_pages; i += gsize) {
      const int pg = P.node_pages[i];
      if (pg < 0 || pg >= P.num_pages) set_status(&hdr->status, SS_ERR_BAD_INPUT);
    }
  }
}

// ---- paths: class, kv length, membership counts of every chain node ------------------------------------------------
__device__ __forceinline__ void plan_paths_phase(const Params& P) {
  PlanHeader* hdr = P.hdr;
  const int live = live_paths(P);
  const int N = P.num_nodes;
  const bool force_generic = (P.flags & SS_FLAG_FORCE_GENERIC) != 0;
  const int64_t gsize = static_cast<int64_t>(gridDim.x) * blockDim.x;
  for (int64_t p64 = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; p64 < live; p64 += gsize) {
    const int p = static_cast<int>(p64);
    const int leaf = P.path_leaf_node[p];
    const int T = P.path_q_len[p];
    bool bad_src = false;
    if (P.q_src_offsets) {
      const int64_t s0 = P.q_src_offsets[p];
      bad_src = s0 < 0 || s0 + T > P.q_src_rows || s0 + T > 0x7fffffffLL;
    }
    if (leaf < 0 || leaf >= N || T < 1 || P.q_offsets[p + 1] - P.q_offsets[p] != T || P.q_offsets[p] < 0 ||
        P.q_offsets[p + 1] > P.total_q || bad_src) {
      set_status(&hdr->status, SS_ERR_BAD_INPUT);
      P.path_class[p] = kClassGeneric;
      continue;
    }
    bool inner_whole_pages = true;
    for (int a = P.node_parent[leaf]; a >= 0; a = P.node_parent[a])
      if (P.node_kv_len[a] % kPage) inner_whole_pages = false;
    int cls;
    if (force_generic) cls = kClassGeneric;
    else if (T == 1) cls = (P.G <= 16) ? kClassDecode : kClassGeneric;
    else cls = inner_whole_pages ? kClassChain : kClassGeneric;
    P.path_class[p] = cls;
    P.path_kv_len[p] = P.node_start[leaf] + P.node_kv_len[leaf];
    if (cls == kClassGeneric) atomicAdd(&hdr->n_generic_rows, T);
    for (int a = leaf; a >= 0; a = P.node_parent[a]) {
      atomicMin(&P.node_first[a], p);
      atomicMax(&P.node_last[a], p);
      atomicAdd(&P.node_npaths[a], 1);
      if (cls == kClassDecode) atomicAdd(&P.node_ndec[a], 1);
    }
  }
}

// ---- every prefix sum -------------------------------------------------------------------------------------------------
__device__ __forceinline__ void plan_scan_phase(const Params& P, int32_t* stage) {   // one whole block; block-uniform
                                                                                     // returns only; stage: see block_excl_scan
  __shared__ int s_total_tiles;
  PlanHeader* hdr = P.hdr;
  if (block_failed(hdr)) return;
  const int tid = threadIdx.x, nt = blockDim.x;
  const int live = live_paths(P);
  const int N = P.num_nodes;
  const int tpt = P.tok_per_tile;
  if (tid == 0) s_total_tiles = 0;

#ifdef SS_STAMPS
  long long pt = clock64();
  int pi = 24;
#define PLAN_MARK() do { __syncthreads(); if (tid == 0) { const long long t = clock64(); hdr->stamp[pi] = t - pt; pt = t; } ++pi; } while (0)
#else
#define PLAN_MARK() do { } while (0)
#endif
  // decode ranks (scanned together with the per-path counts below where one pass can take all four arrays)
  const bool fused = live <= nt * kScanRegs &&
                     ((reinterpret_cast<uintptr_t>(P.path_slot_base) | reinterpret_cast<uintptr_t>(P.path_leaf_base) |
                       reinterpret_cast<uintptr_t>(P.path_chain_base) | reinterpret_cast<uintptr_t>(P.path_dec_rank)) & 15) == 0;
  for (int p = tid; p < live; p += nt) P.path_dec_rank[p] = (P.path_class[p] == kClassDecode) ? 1 : 0;
  if (!fused) {
    const int n_dec = block_excl_scan(P.path_dec_rank, live, stage);
    if (tid == 0) {
      P.path_dec_rank[live] = n_dec;
      hdr->n_dec = n_dec;
      if (n_dec > P.caps.dec) set_status(&hdr->status, SS_ERR_WORKSPACE_TOO_SMALL);
    }
  }

  PLAN_MARK();   // 8: decode ranks
  // nodes: role, tiles
  for (int n = tid; n < N; n += nt) {
    const int np = P.node_npaths[n];
    if (np > 0 && P.node_last[n] - P.node_first[n] + 1 != np) set_status(&hdr->status, SS_ERR_BAD_INPUT);
    const int nd = P.node_ndec[n], len = P.node_kv_len[n];
    int tiles = 0;
    if (nd > 0 && len > 0) {
      const bool leaf_only = (np == 1 && P.path_leaf_node[P.node_first[n]] == n);
      if (!leaf_only) tiles = ceil_div(nd, tpt);
    }
    P.node_item_base[n] = tiles;                     // tiles for now; becomes the item base after the scan
    if (tiles) atomicAdd(&s_total_tiles, tiles);
  }
  if (block_failed(hdr)) return;
  PLAN_MARK();   // 9: node tiles
  const int total_tiles = s_total_tiles * P.Hkv;
  for (int n = tid; n < N; n += nt) {
    const int nd = P.node_ndec[n], len = P.node_kv_len[n];
    const int tiles = P.node_item_base[n];
    int splits = 1, own = 0, split_len = len;
    if (nd > 0 && len > 0) {
      if (tiles == 0) {
        own = ceil_div(len, kLeafChunk);             // private leaf of one decode path
      } else {
        if (P.node_depth[n] == 0) node_split(P, len, total_tiles, splits, split_len);
        own = splits;
      }
    }
    P.node_splits[n] = splits;
    P.node_split_len[n] = split_len;
    P.node_own_slots[n] = own;
    P.node_item_base[n] = tiles * splits * P.Hkv;
  }
  __syncthreads();
  PLAN_MARK();   // 10: splits
  for (int n = tid; n < N; n += nt) {
    int off = 0;
    for (int a = P.node_parent[n]; a >= 0; a = P.node_parent[a]) off += P.node_own_slots[a];
    P.node_level_off[n] = off;
  }
  PLAN_MARK();   // 11: level offsets
  const int n_stacked = block_excl_scan(P.node_item_base, N, stage);
  PLAN_MARK();   // 12: item base scan
  if (tid == 0) P.node_item_base[N] = n_stacked;

  // decode paths: partial slots, leaf items; chain paths: tile items
  for (int p = tid; p < live; p += nt) {
    int slots = 0, leaf_items = 0, chain_items = 0;
    const int cls = P.path_class[p];
    if (cls == kClassDecode) {
      const int leaf = P.path_leaf_node[p];
      slots = P.node_level_off[leaf] + P.node_own_slots[leaf];
      if (P.node_npaths[leaf] == 1 && P.node_kv_len[leaf] > 0)
        leaf_items = ceil_div(P.node_kv_len[leaf], kLeafChunk) * P.Hkv;
    } else if (cls == kClassChain) {
      chain_items = ceil_div(P.path_q_len[p], tpt) * P.Hkv;
    }
    P.path_slot_base[p] = slots;
    P.path_leaf_base[p] = leaf_items;
    P.path_chain_base[p] = chain_items;
  }
  PLAN_MARK();   // 13: per-path counts
  int n_slots, n_leaf_items, n_chain;
  if (fused) {
    int t2[2];
    block_excl_scan2_regs(P.path_slot_base, P.path_leaf_base, live, t2);
    n_slots = t2[0];
    n_leaf_items = t2[1];
    block_excl_scan2_regs(P.path_chain_base, P.path_dec_rank, live, t2);
    n_chain = t2[0];
    if (tid == 0) {
      P.path_dec_rank[live] = t2[1];
      hdr->n_dec = t2[1];
      if (t2[1] > P.caps.dec) set_status(&hdr->status, SS_ERR_WORKSPACE_TOO_SMALL);
    }
  } else {
    n_slots = block_excl_scan(P.path_slot_base, live, stage);
    n_leaf_items = block_excl_scan(P.path_leaf_base, live, stage);
    n_chain = block_excl_scan(P.path_chain_base, live, stage);
  }
  PLAN_MARK();   // 14: three scans
  if (tid == 0) {
    hdr->n_slots = n_slots;
    hdr->n_stacked_items = n_stacked;
    if (n_slots > P.caps.slots || n_leaf_items > P.caps.leaf_items || n_stacked + n_chain > P.caps.tile_items) {
      set_status(&hdr->status, SS_ERR_WORKSPACE_TOO_SMALL);     // the executors see the status and do nothing
    } else {
      hdr->n_leaf_items = n_leaf_items;
      hdr->n_tile_items = n_stacked + n_chain;
    }
  }
}

// ---- item lists ---------------------------------------------------------------------------------------------------------
__device__ __forceinline__ void plan_emit_phase(const Params& P) {
  PlanHeader* hdr = P.hdr;
  const int live = live_paths(P);
  const int N = P.num_nodes;
  const int tpt = P.tok_per_tile;
  const int n_stacked = hdr->n_stacked_items;
  const int64_t gtid = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  const int64_t gsize = static_cast<int64_t>(gridDim.x) * blockDim.x;
  if (gtid == 0) P.dec_slot_base[hdr->n_dec] = hdr->n_slots;

  // per decode token: output row, query row, partial slots, leaf chunks, arrival counters
  for (int64_t p64 = gtid; p64 < live; p64 += gsize) {
    const int p = static_cast<int>(p64);
    if (P.path_class[p] != kClassDecode) continue;
    const int rank = P.path_dec_rank[p];
    const int leaf = P.path_leaf_node[p];
    const int len = P.node_kv_len[leaf];
    P.dec_tok[rank] = static_cast<int32_t>(P.q_offsets[p]);
    P.dec_src[rank] = static_cast<int32_t>(P.q_src_offsets ? P.q_src_offsets[p] : P.q_offsets[p]);
    P.dec_slot_base[rank] = P.path_slot_base[p];
    const bool own_leaf = P.node_npaths[leaf] == 1 && len > 0;
    P.dec_leaf_chunks[rank] = own_leaf ? ceil_div(len, kLeafChunk) : 0;
    for (int g = 0; g < P.Hkv; ++g) P.leaf_arrive[static_cast<int64_t>(rank) * P.Hkv + g] = 0;
  }
  // Leaf and chain items, one thread per ITEM (consecutive threads write consecutive descriptors: a thread per path
  // writing its own run of descriptors makes every store instruction touch 32 different sectors, and that alone cost
  // tens of microseconds on one SM).  Item e -> path by binary search over the exclusive scans.
  auto path_of = [&](const int32_t* base, int e) {
    int lo = 0, hi = live;                    // last p with base[p] <= e (paths without items share their successor's base)
    while (hi - lo > 1) {
      const int mid = (lo + hi) >> 1;
      if (base[mid] <= e) lo = mid; else hi = mid;
    }
    return lo;
  };
  const int n_leaf_items = hdr->n_leaf_items;
  for (int64_t e64 = gtid; e64 < n_leaf_items; e64 += gsize) {
    const int e = static_cast<int>(e64);
    const int p = path_of(P.path_leaf_base, e);
    const int local = e - P.path_leaf_base[p];
    const int c = local / P.Hkv, g = local - c * P.Hkv;
    const int leaf = P.path_leaf_node[p];
    const int len = P.node_kv_len[leaf];
    LeafItem it;
    it.page0 = static_cast<int32_t>(P.node_page_offsets[leaf]) + c * (kLeafChunk / kPage);
    it.node = leaf;
    it.g = g;
    it.kv_begin = c * kLeafChunk;
    it.kv_end = min(len, (c + 1) * kLeafChunk);
    it.slot = P.path_slot_base[p] + P.node_level_off[leaf] + c;
    it.q_src = static_cast<int32_t>(P.q_src_offsets ? P.q_src_offsets[p] : P.q_offsets[p]);
    it.dec = P.path_dec_rank[p];
    P.leaf_items[e] = it;
  }
  const int n_chain_items = hdr->n_tile_items - n_stacked;
  for (int64_t e64 = gtid; e64 < n_chain_items; e64 += gsize) {
    const int e = static_cast<int>(e64);
    const int p = path_of(P.path_chain_base, e);
    const int local = e - P.path_chain_base[p];
    const int T = P.path_q_len[p];
    const int L = P.path_kv_len[p];
    const int tiles = ceil_div(T, tpt);
    const int g = local / tiles, t = local - g * tiles;
    const int32_t src_row = static_cast<int32_t>(P.q_src_offsets ? P.q_src_offsets[p] : P.q_offsets[p]);
    TileItem it;
    it.node = P.path_leaf_node[p];
    it.tok0 = static_cast<int32_t>(P.q_offsets[p]) + t * tpt;
    it.n_tok = min(tpt, T - t * tpt);
    it.kind_g = (kItemChain << 16) | g;
    it.kv_begin = 0;
    it.limit0 = L - T + t * tpt + 1;
    it.kv_end = max(0, min(L, it.limit0 + it.n_tok - 1));
    it.slot_off = -1;
    it.src0 = src_row + t * tpt;
    it.pad = 0;
    P.tile_items[n_stacked + e] = it;
  }

  // stacked items: item e -> node by binary search over the exclusive scan of per-node item counts
  for (int64_t e64 = gtid; e64 < n_stacked; e64 += gsize) {
    const int e = static_cast<int>(e64);
    int lo = 0, hi = N;                       // last n with base[n] <= e and base[n+1] > e
    while (hi - lo > 1) {
      const int mid = (lo + hi) >> 1;
      if (P.node_item_base[mid] <= e) lo = mid; else hi = mid;
    }
    const int n = lo;
    const int local = e - P.node_item_base[n];
    const int splits = P.node_splits[n];
    const int split = local % splits;
    const int rest = local / splits;
    const int g = rest % P.Hkv;
    const int tile = rest / P.Hkv;
    const int len = P.node_kv_len[n];
    const int split_len = P.node_split_len[n];
    const int nd = P.node_ndec[n];
    TileItem it;
    it.node = n;
    it.tok0 = P.path_dec_rank[P.node_first[n]] + tile * tpt;
    it.n_tok = min(tpt, nd - tile * tpt);
    it.kind_g = (kItemStacked << 16) | g;
    it.kv_begin = split * split_len;
    it.kv_end = min(len, (split + 1) * split_len);
    it.limit0 = it.kv_end;
    it.slot_off = P.node_level_off[n] + split;
    it.src0 = static_cast<int32_t>(P.node_page_offsets[n]);
    it.pad = 0;
    P.tile_items[e] = it;
  }
}

// ---- general path: four launches ------------------------------------------------------------------------------------
__global__ void __launch_bounds__(kGridThreads) plan_nodes_kernel(const Params P) {
  ss::grid_dependency_enter();
  plan_nodes_phase(P);
}
__global__ void __launch_bounds__(kGridThreads) plan_paths_kernel(const Params P) {
  ss::grid_dependency_enter();
  if (P.hdr->status != SS_OK) return;          // no barrier in this kernel: a per-thread return is safe
  plan_paths_phase(P);
}
__global__ void __launch_bounds__(kScanThreads) plan_scan_kernel(const Params P) {
  ss::grid_dependency_enter();
  extern __shared__ __align__(16) int32_t scan_stage[];
  plan_scan_phase(P, scan_stage);
}
__global__ void __launch_bounds__(kGridThreads) plan_emit_kernel(const Params P) {
  ss::grid_dependency_enter();
  if (P.hdr->status != SS_OK) return;          // no barrier in this kernel
  plan_emit_phase(P);
}

// ---- small trees: one launch, everything in shared memory ---------------------------------------------------------
constexpr int kSmallPlan = 2048;               // nodes and paths: two of each per thread
constexpr int kSmallNodeArrays = 14, kSmallPathArrays = 10;
inline size_t small_plan_smem(int N, int NP) {
  return static_cast<size_t>(4) * (static_cast<size_t>(N) * kSmallNodeArrays + static_cast<size_t>(NP) * kSmallPathArrays) + 64;
}
// Blocks: what is left to share is the emission, a warp per path and per node.
inline int small_plan_blocks(int N, int NP) {
  const int b = (N + NP + 31) / 32;
  return b < 1 ? 1 : (b > 64 ? 64 : b);
}
constexpr int kLeafClasses = 17;               // pages of the last chunk of a leaf: 0 .. 16

// Six exclusive scans at once over the block's entries 2 tid, 2 tid + 1 (v -> positions), and the totals; in the same two
// barriers the rank of each entry among all of them, larger classes cls[] first (order[]: deterministic, but not index
// order within a class).
struct SmallScan {
  int tot[6][32];              // per warp, then exclusive over the warps
  int total[6];
  int hist[kLeafClasses][64];  // per class and group of 32 entries, then exclusive over the groups
  int cls_total[kLeafClasses];
};
__device__ __forceinline__ void small_scan(SmallScan& S, int (&v)[6][2], const int (&cls)[2], int (&order)[2]) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  int sum[6], x[6];
#pragma unroll
  for (int k = 0; k < 6; ++k) x[k] = sum[k] = v[k][0] + v[k][1];
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
#pragma unroll
    for (int k = 0; k < 6; ++k) {
      const int y = __shfl_up_sync(0xffffffffu, x[k], o);
      if (lane >= o) x[k] += y;
    }
  }
  if (lane == 31) {
#pragma unroll
    for (int k = 0; k < 6; ++k) S.tot[k][warp] = x[k];
  }
  int in_group[2];
#pragma unroll
  for (int e = 0; e < 2; ++e) {
    const uint32_t peers = __match_any_sync(0xffffffffu, cls[e]);
    in_group[e] = __popc(peers & ((1u << lane) - 1u));
    if (in_group[e] == 0) S.hist[cls[e]][2 * warp + e] = __popc(peers);   // (the rest was cleared by the caller)
  }
  __syncthreads();
  if (warp < 6) {
    const int t = S.tot[warp][lane];
    int y = t;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int z = __shfl_up_sync(0xffffffffu, y, o);
      if (lane >= o) y += z;
    }
    S.tot[warp][lane] = y - t;
    if (lane == 31) S.total[warp] = y;
  } else if (warp >= 8 && warp < 8 + kLeafClasses) {
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
  for (int k = 0; k < 6; ++k) {
    const int first = S.tot[k][warp] + x[k] - sum[k];
    v[k][1] = first + v[k][0];
    v[k][0] = first;
  }
  int above = lane < kLeafClasses ? S.cls_total[lane] : 0;      // lane r: entries of the classes > r
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

__global__ void __launch_bounds__(kScanThreads) plan_small_kernel(const __grid_constant__ Params P) {
  ss::grid_dependency_enter();
  extern __shared__ __align__(16) int32_t plan_smem[];
  __shared__ PlanHeader s_hdr;
  __shared__ SmallScan s_scan;
  __shared__ int s_total_tiles, s_generic;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int N = P.num_nodes, NP = P.num_paths, Hkv = P.Hkv, tpt = P.tok_per_tile;
  int32_t* w = plan_smem;
  auto take = [&](int n) { int32_t* r = w; w += n; return r; };
  int32_t *n_parent = take(N), *n_len = take(N), *n_page0 = take(N), *n_start = take(N), *n_first = take(N), *n_last = take(N),
          *n_paths = take(N), *n_dec = take(N), *n_own = take(N), *n_level = take(N), *n_tiles = take(N), *n_splits = take(N),
          *n_split_len = take(N), *n_base = take(N);
  int32_t *p_leaf = take(NP), *p_T = take(NP), *p_row = take(NP), *p_src = take(NP), *p_class = take(NP), *p_rank = take(NP),
          *p_slot = take(NP), *p_full = take(NP), *p_chain = take(NP), *p_last = take(NP);

  for (int x = tid; x < static_cast<int>(sizeof(PlanHeader) / 4); x += kScanThreads) reinterpret_cast<int32_t*>(&s_hdr)[x] = 0;
  for (int x = tid; x < kLeafClasses * 64; x += kScanThreads) (&s_scan.hist[0][0])[x] = 0;
  if (tid == 0) s_total_tiles = s_generic = 0;
  SS_STAMP_BEGIN(P.hdr, 0);

  // ---- inputs (one trip: the per-path arrays are read up to their capacity, beside the live count) -----------------------
  const int live = live_paths(P);
  bool bad = false;
#pragma unroll 1
  for (int i = tid; i < max(N, NP); i += kScanThreads) {       // (node i and path i: their loads go out together)
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
      n_parent[n] = parent;
      n_len[n] = len;
      n_page0[n] = static_cast<int32_t>(o0);
      n_first[n] = 0x7fffffff;
      n_last[n] = -1;
      n_paths[n] = n_dec[n] = 0;
    }
    if (i < NP) {
      bool ok = leaf >= 0 && leaf < N && T >= 1 && r1 - r0 == T && r0 >= 0 && r1 <= P.total_q;
      if (P.q_src_offsets) ok = ok && src >= 0 && src + T <= P.q_src_rows && src + T <= 0x7fffffffLL;
      p_leaf[p] = ok ? leaf : -1;
      p_T[p] = T;
      p_row[p] = static_cast<int32_t>(r0);
      p_src[p] = static_cast<int32_t>(src);
    }
  }
  if (P.flags & SS_FLAG_VALIDATE) {
    for (int64_t i = tid; i < P.total_node_pages; i += kScanThreads) {
      const int pg = P.node_pages[i];
      bad = bad || pg < 0 || pg >= P.num_pages;
    }
  }
  bool failed = __syncthreads_or(bad) != 0;
  if (failed && tid == 0) s_hdr.status = SS_ERR_BAD_INPUT;

  // ---- nodes: keys before the node (parents come first, so every walk ends) -------------------------------------------------
  if (!failed) {
    bool deep = false;
#pragma unroll 1
    for (int n = tid; n < N; n += kScanThreads) {
      int d = 1, start = 0;
#pragma unroll 1
      for (int a = n_parent[n]; a >= 0 && d <= SS_MAX_DEPTH; a = n_parent[a]) { start += n_len[a]; ++d; }
      deep = deep || d > SS_MAX_DEPTH;
      n_start[n] = start;
    }
    failed = __syncthreads_or(deep) != 0;
    if (failed && tid == 0) s_hdr.status = SS_ERR_UNSUPPORTED;
  }

  // ---- paths: class, membership of every chain node (lanes with the same node are counted together) ---------------------
  if (!failed) {
    bad = false;
#pragma unroll 1
    for (int p0 = 0; p0 < live; p0 += kScanThreads) {
      const int p = p0 + tid;
      const int leaf = p < live ? p_leaf[p] : -1, T = p < live ? p_T[p] : 0;
      bad = bad || (p < live && leaf < 0);
      const bool force = (P.flags & SS_FLAG_FORCE_GENERIC) != 0;
      const bool dec = leaf >= 0 && T == 1 && P.G <= 16 && !force;
      const uint32_t decs = __ballot_sync(0xffffffffu, dec);
      bool whole = true;                                       // inner nodes are whole pages
      int a = leaf;
#pragma unroll 1
      while (__any_sync(0xffffffffu, a >= 0)) {
        const uint32_t peers = __match_any_sync(0xffffffffu, a);
        if (a >= 0) {
          if ((peers & ((1u << lane) - 1u)) == 0) {
            atomicMin(&n_first[a], p);
            atomicMax(&n_last[a], p + 31 - __clz(peers) - lane);
            atomicAdd(&n_paths[a], __popc(peers));
            if (peers & decs) atomicAdd(&n_dec[a], __popc(peers & decs));
          }
          if (a != leaf && n_len[a] % kPage) whole = false;
          a = n_parent[a];
        }
      }
      if (leaf >= 0) {
        const int cls = dec ? kClassDecode : (force || T == 1 || !whole ? kClassGeneric : kClassChain);
        p_class[p] = cls;
        if (cls == kClassGeneric) atomicAdd(&s_generic, T);
      }
    }
    failed = __syncthreads_or(bad) != 0;
    if (failed && tid == 0) s_hdr.status = SS_ERR_BAD_INPUT;
  }

  // ---- nodes: tiles ----------------------------------------------------------------------------------------------------
  if (!failed) {
    bad = false;
    int mine = 0;
#pragma unroll 1
    for (int n = tid; n < N; n += kScanThreads) {
      const int np = n_paths[n], nd = n_dec[n];
      bad = bad || (np > 0 && n_last[n] - n_first[n] + 1 != np);
      int tiles = 0;
      if (nd > 0 && n_len[n] > 0 && !(np == 1 && p_leaf[n_first[n]] == n)) tiles = ceil_div(nd, tpt);
      n_tiles[n] = tiles;
      mine += tiles;
    }
    mine = static_cast<int>(__reduce_add_sync(0xffffffffu, static_cast<unsigned>(mine)));
    if (lane == 0 && mine) atomicAdd(&s_total_tiles, mine);
    failed = __syncthreads_or(bad) != 0;
    if (failed && tid == 0) s_hdr.status = SS_ERR_BAD_INPUT;
  }

  // ---- nodes: KV splits, partial slots -----------------------------------------------------------------------------------
  if (!failed) {
    const int total_tiles = s_total_tiles * Hkv;
#pragma unroll 1
    for (int n = tid; n < N; n += kScanThreads) {
      const int len = n_len[n], tiles = n_tiles[n];
      int splits = 1, own = 0, split_len = len;
      if (tiles > 0) {
        if (n_parent[n] < 0) node_split(P, len, total_tiles, splits, split_len);
        own = splits;
      } else if (n_dec[n] > 0 && len > 0) {
        own = ceil_div(len, kLeafChunk);                     // private leaf of one decode path
      }
      n_splits[n] = splits;
      n_split_len[n] = split_len;
      n_own[n] = own;
    }
    __syncthreads();

    // ---- every prefix sum: entries 2 tid, 2 tid + 1 of the nodes and of the paths ------------------------------------------
    int v[6][2], cls[2] = {0, 0}, order[2];
#pragma unroll 1
    for (int e = 0; e < 2; ++e) {
      const int i = 2 * tid + e;
      int root_items = 0, node_items = 0, slots = 0, full = 0, chain = 0, dec = 0, c = 0;
      if (i < N) {
        int off = 0;
#pragma unroll 1
        for (int a = n_parent[i]; a >= 0; a = n_parent[a]) off += n_own[a];
        n_level[i] = off;
        const int items = n_tiles[i] * n_splits[i] * Hkv;
        if (n_parent[i] < 0) root_items = items; else node_items = items;
      }
      if (i < live) {
        const int leaf = p_leaf[i], len = n_len[leaf];
        if (p_class[i] == kClassDecode) {
          dec = 1;
#pragma unroll 1
          for (int a = leaf; a >= 0; a = n_parent[a]) slots += n_own[a];
          if (n_paths[leaf] == 1 && len > 0) {
            full = len / kLeafChunk;
            c = ceil_div(len - full * kLeafChunk, kPage);
          }
        } else if (p_class[i] == kClassChain) {
          chain = ceil_div(p_T[i], tpt) * Hkv;
        }
      }
      if (e == 0) {
        v[0][0] = root_items; v[1][0] = node_items; v[2][0] = dec; v[3][0] = slots; v[4][0] = full; v[5][0] = chain; cls[0] = c;
      } else {
        v[0][1] = root_items; v[1][1] = node_items; v[2][1] = dec; v[3][1] = slots; v[4][1] = full; v[5][1] = chain; cls[1] = c;
      }
    }
    small_scan(s_scan, v, cls, order);
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const int i = 2 * tid + e;
      if (i < N) n_base[i] = n_parent[i] < 0 ? v[0][e] : s_scan.total[0] + v[1][e];   // the roots' items come first
      if (i < live) {
        p_rank[i] = v[2][e];
        p_slot[i] = v[3][e];
        p_full[i] = v[4][e];
        p_chain[i] = v[5][e];
        p_last[i] = cls[e] > 0 ? order[e] : -1;
      }
    }
    __syncthreads();
  }

  if (!failed) {
    const int n_stacked = s_scan.total[0] + s_scan.total[1], n_dec_tok = s_scan.total[2], n_slots = s_scan.total[3];
    const int n_full = s_scan.total[4] * Hkv, n_chain = s_scan.total[5];
    int n_last_chunks = 0;
    for (int r = 1; r < kLeafClasses; ++r) n_last_chunks += s_scan.cls_total[r];
    const int n_leaf_items = n_full + n_last_chunks * Hkv;
    failed = n_dec_tok > P.caps.dec || n_slots > P.caps.slots || n_leaf_items > P.caps.leaf_items || n_stacked + n_chain > P.caps.tile_items;
    if (tid == 0) {
      s_hdr.status = failed ? SS_ERR_WORKSPACE_TOO_SMALL : SS_OK;
      s_hdr.n_dec = n_dec_tok;
      s_hdr.n_slots = n_slots;
      s_hdr.n_stacked_items = n_stacked;
      s_hdr.n_generic_rows = s_generic;
      if (!failed) {
        s_hdr.n_leaf_items = n_leaf_items;
        s_hdr.n_tile_items = n_stacked + n_chain;
      }
    }
    if (!failed) {
      // ---- emission: a warp per path and per node --------------------------------------------------------------------------
      const int wid = blockIdx.x * (kScanThreads / 32) + warp, nw = gridDim.x * (kScanThreads / 32);
      if (wid == 0 && lane == 0) P.dec_slot_base[n_dec_tok] = n_slots;
#pragma unroll 1
      for (int p = wid; p < live; p += nw) {
        const int leaf = p_leaf[p], len = n_len[leaf], cls = p_class[p], L = n_start[leaf] + len;
        if (lane == 0) {                                       // (read by the generic rows and the exact second pass)
          P.path_class[p] = cls;
          P.path_kv_len[p] = L;
        }
        if (cls == kClassDecode) {
          const int rank = p_rank[p], slot = p_slot[p];
          const bool own_leaf = n_paths[leaf] == 1 && len > 0;
          if (lane == 0) {
            P.dec_tok[rank] = p_row[p];
            P.dec_src[rank] = p_src[p];
            P.dec_slot_base[rank] = slot;
            P.dec_leaf_chunks[rank] = own_leaf ? ceil_div(len, kLeafChunk) : 0;
          }
          for (int g = lane; g < Hkv; g += 32) P.leaf_arrive[static_cast<int64_t>(rank) * Hkv + g] = 0;
          if (!own_leaf) continue;
          // whole chunks first, then the last chunks of all leaves, longest first: the leaf kernel hands its items out in
          // this order, and the short ones level out its warps' ends (922 leaves of 32 to 512 keys: 71.6 -> 68.9 us)
          const int full = len / kLeafChunk, last = p_last[p], n_items = (full + (last >= 0 ? 1 : 0)) * Hkv;
#pragma unroll 1
          for (int x = lane; x < n_items; x += 32) {
            const int c = x / Hkv, g = x - c * Hkv;
            LeafItem it;
            it.page0 = n_page0[leaf] + c * (kLeafChunk / kPage);
            it.node = leaf;
            it.g = g;
            it.kv_begin = c * kLeafChunk;
            it.kv_end = min(len, (c + 1) * kLeafChunk);
            it.slot = slot + n_level[leaf] + c;
            it.q_src = p_src[p];
            it.dec = rank;
            P.leaf_items[c < full ? p_full[p] * Hkv + x : n_full + last * Hkv + g] = it;
          }
        } else if (cls == kClassChain) {
          const int T = p_T[p], tiles = ceil_div(T, tpt);
#pragma unroll 1
          for (int x = lane; x < tiles * Hkv; x += 32) {
            const int g = x / tiles, t = x - g * tiles;
            TileItem it;
            it.node = leaf;
            it.tok0 = p_row[p] + t * tpt;
            it.n_tok = min(tpt, T - t * tpt);
            it.kind_g = (kItemChain << 16) | g;
            it.kv_begin = 0;
            it.limit0 = L - T + t * tpt + 1;
            it.kv_end = max(0, min(L, it.limit0 + it.n_tok - 1));
            it.slot_off = -1;
            it.src0 = p_src[p] + t * tpt;
            it.pad = 0;
            P.tile_items[n_stacked + p_chain[p] + x] = it;
          }
        }
      }
#pragma unroll 1
      for (int n = wid; n < N; n += nw) {
        if (lane == 0) P.node_start[n] = n_start[n];
        const int tiles = n_tiles[n];
        if (tiles == 0) continue;
        const int splits = n_splits[n], split_len = n_split_len[n], len = n_len[n], nd = n_dec[n], rank0 = p_rank[n_first[n]];
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
          it.slot_off = n_level[n] + split;
          it.src0 = n_page0[n];
          it.pad = 0;
          P.tile_items[n_base[n] + x] = it;
        }
      }
    }
  }
  if (blockIdx.x != 0) return;
  if (tid == 0) s_hdr.live_paths = live;
#ifdef SS_STAMPS
  __syncthreads();
  if (tid == 0) { s_hdr.stamp[0] = P.hdr->stamp[0]; s_hdr.stamp[1] = ss_globaltimer(); }
#endif
  __syncthreads();
  for (int x = tid; x < static_cast<int>(sizeof(PlanHeader) / 4); x += kScanThreads)
    reinterpret_cast<int32_t*>(P.hdr)[x] = reinterpret_cast<const int32_t*>(&s_hdr)[x];
}

int32_t launch_plan(const Params& P, cudaStream_t st) {
  if (P.num_nodes <= kSmallPlan && P.num_paths <= kSmallPlan) {     // (this kernel writes the whole header itself)
    static bool configured[kDeviceSlots] = {false};
    const int dev_slot = current_device_slot();
    if (dev_slot < 0 || !configured[dev_slot]) {
      if (cudaFuncSetAttribute(plan_small_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               static_cast<int>(small_plan_smem(kSmallPlan, kSmallPlan))) != cudaSuccess) {
        (void)cudaGetLastError();
        return SS_ERR_CUDA;
      }
      if (dev_slot >= 0) configured[dev_slot] = true;
    }
    SS_LAUNCH(plan_small_kernel, small_plan_blocks(P.num_nodes, P.num_paths), kScanThreads,
              small_plan_smem(P.num_nodes, P.num_paths), st, P);
    return SS_OK;
  }
  if (cudaMemsetAsync(P.hdr, 0, sizeof(PlanHeader), st) != cudaSuccess) {
    (void)cudaGetLastError();
    return SS_ERR_CUDA;
  }
  const int64_t work = P.num_nodes > P.num_paths ? P.num_nodes : P.num_paths;
  int blocks = static_cast<int>((work + kGridThreads - 1) / kGridThreads);
  if (blocks < 1) blocks = 1;
  if (blocks > 1184) blocks = 1184;
  SS_LAUNCH(plan_nodes_kernel, blocks, kGridThreads, 0, st, P);
  SS_LAUNCH(plan_paths_kernel, blocks, kGridThreads, 0, st, P);
  {
    static bool configured[kDeviceSlots] = {false};
    const int dev_slot = current_device_slot();
    if (dev_slot < 0 || !configured[dev_slot]) {
      if (cudaFuncSetAttribute(plan_scan_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kScanStage * 4) != cudaSuccess) {
        (void)cudaGetLastError();
        return SS_ERR_CUDA;
      }
      if (dev_slot >= 0) configured[dev_slot] = true;
    }
  }
  SS_LAUNCH(plan_scan_kernel, 1, kScanThreads, kScanStage * 4, st, P);
  // one thread per ITEM (there are an order of magnitude more items than paths; their number is known on the device
  // only): a grid that covers the typical item count in one or two strides
  SS_LAUNCH(plan_emit_kernel, blocks < 64 ? 8 * blocks : 1184, kGridThreads, 0, st, P);
  return SS_OK;
}

}  // namespace attn
}  // namespace ss
