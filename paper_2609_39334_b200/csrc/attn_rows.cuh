// One query row per warp, keys visited one at a time with an online softmax, all in fp32: lane l owns dims 4l..4l+3
// of q and of the output accumulator.  Shared by the plain kernels (attn_simple.cu) and by the exact second pass of
// the tensor-core tile kernel (a tile item whose scores left the range of its lagged reference maximum).
#pragma once
#include "attn_plan.cuh"

namespace ss {
namespace attn {

struct RowState {
  float q[4];
  float acc[4];
  float m, l;
};

__device__ __forceinline__ void load4(const __nv_bfloat16* p, float (&v)[4]) {
  const uint2 u = *reinterpret_cast<const uint2*>(p);
  const __nv_bfloat162 a = *reinterpret_cast<const __nv_bfloat162*>(&u.x);
  const __nv_bfloat162 b = *reinterpret_cast<const __nv_bfloat162*>(&u.y);
  v[0] = __low2float(a); v[1] = __high2float(a); v[2] = __low2float(b); v[3] = __high2float(b);
}

__device__ __forceinline__ void row_init(RowState& r, const __nv_bfloat16* qrow, int lane) {
  load4(qrow + 4 * lane, r.q);
  r.acc[0] = r.acc[1] = r.acc[2] = r.acc[3] = 0.f;
  r.m = -INFINITY;
  r.l = 0.f;
}

// Visit keys [t0, t1) of one node (t relative to the node).
__device__ __forceinline__ void row_visit_node(RowState& r, const Params& P, int node, int g, int t0, int t1, int lane) {
  if (t1 <= t0) return;
  const int64_t pg0 = P.node_page_offsets[node];
  for (int t = t0; t < t1; ++t) {
    int64_t page = P.node_pages[pg0 + t / kPage];
    SS_CHECK_OR(page >= 0 && page < P.num_pages, &P.hdr->status, page = 0);
    const int64_t off = page * P.page_stride + static_cast<int64_t>(g) * P.head_stride +
                        static_cast<int64_t>(t % kPage) * P.token_stride + 4 * lane;
    float k[4], v[4];
    load4(P.k_pool + off, k);
    float s = r.q[0] * k[0] + r.q[1] * k[1] + r.q[2] * k[2] + r.q[3] * k[3];
    s = warp_sum(s) * P.scale;
    load4(P.v_pool + off, v);
    const float m_new = fmaxf(r.m, s);
    const float corr = __expf(r.m - m_new);          // exp(-inf) = 0 on the first key
    const float p = __expf(s - m_new);
    r.l = r.l * corr + p;
#pragma unroll
    for (int i = 0; i < 4; ++i) r.acc[i] = r.acc[i] * corr + p * v[i];
    r.m = m_new;
  }
}

__device__ __forceinline__ void row_store_final(const RowState& r, const Params& P, int64_t q_row, int h, int lane) {
  const float inv = r.l > 0.f ? 1.f / r.l : 0.f;
  __nv_bfloat16* o = P.out + (q_row * P.Hq + h) * kHeadDim + 4 * lane;
  __nv_bfloat162 a = __floats2bfloat162_rn(r.acc[0] * inv, r.acc[1] * inv);
  __nv_bfloat162 b = __floats2bfloat162_rn(r.acc[2] * inv, r.acc[3] * inv);
  uint2 u;
  u.x = *reinterpret_cast<uint32_t*>(&a);
  u.y = *reinterpret_cast<uint32_t*>(&b);
  *reinterpret_cast<uint2*>(o) = u;
  if (P.lse && lane == 0) P.lse[q_row * P.Hq + h] = r.l > 0.f ? r.m + __logf(r.l) : -INFINITY;
}

__device__ __forceinline__ void row_store_partial(const RowState& r, const Params& P, int64_t slot, int h, int lane) {
  const float inv = r.l > 0.f ? 1.f / r.l : 0.f;
  float4 o = make_float4(r.acc[0] * inv, r.acc[1] * inv, r.acc[2] * inv, r.acc[3] * inv);
  *reinterpret_cast<float4*>(P.part_o + (slot * P.Hq + h) * kHeadDim + 4 * lane) = o;
  if (lane == 0) P.part_lse[slot * P.Hq + h] = r.l > 0.f ? r.m + __logf(r.l) : -INFINITY;
}

// Keys [v0, v1) of the virtual sequence root -> `leaf` (chain nodes concatenated).
__device__ inline void row_visit_chain(RowState& r, const Params& P, int leaf, int g, int v0, int v1, int lane) {
  int chain[SS_MAX_DEPTH];
  int d = 0;
  for (int a = leaf; a >= 0 && d < SS_MAX_DEPTH; a = P.node_parent[a]) chain[d++] = a;
  for (int c = d - 1; c >= 0; --c) {
    const int n = chain[c];
    const int start = P.node_start[n], len = P.node_kv_len[n];
    const int t0 = max(v0 - start, 0), t1 = min(v1 - start, len);
    row_visit_node(r, P, n, g, t0, t1, lane);
  }
}

// One tile item, exactly: rows `warp_index`, `warp_index + n_warps`, ... of the item, one warp each (whole warps).
__device__ __forceinline__ void tile_item_rows_exact(const Params& P, const TileItem& it, int warp_index, int n_warps, int lane) {
  const int kind = it.kind_g >> 16, g = it.kind_g & 0xffff;
  const int rows = it.n_tok * P.G;
  for (int rrow = warp_index; rrow < rows; rrow += n_warps) {
    const int i = rrow / P.G, h = g * P.G + rrow % P.G;
    const int dec = it.tok0 + i;                       // stacked: index into dec_tok
    const int64_t q_row = (kind == kItemChain) ? static_cast<int64_t>(it.tok0 + i) : P.dec_tok[dec];
    const int64_t q_src = (kind == kItemChain) ? static_cast<int64_t>(it.src0 + i) : P.dec_src[dec];
    const int visible = (kind == kItemChain) ? it.limit0 + i : it.limit0;
    const int v1 = min(it.kv_end, visible);
    RowState r;
    row_init(r, P.q + (q_src * P.Hq + h) * kHeadDim, lane);
    if (kind == kItemChain) {
      row_visit_chain(r, P, it.node, g, it.kv_begin, v1, lane);
      row_store_final(r, P, q_row, h, lane);
    } else {
      row_visit_node(r, P, it.node, g, it.kv_begin, v1, lane);
      row_store_partial(r, P, static_cast<int64_t>(P.dec_slot_base[dec]) + it.slot_off, h, lane);
    }
  }
}

// Log-sum-exp merge of the per-level partial results of decode token `d`, q head `h` (one whole warp):
// out = sum_s exp(lse_s - LSE) o_s,  LSE = log sum_s exp(lse_s); a token without partials (no keys) gives 0 / -inf.
// The partials are read from L2 (ld.global.cg): inside the leaf kernel they may have been written by other SMs
// moments ago.
__device__ __forceinline__ void merge_row(const Params& P, int d, int h, int lane) {
  const int s0 = P.dec_slot_base[d], s1 = P.dec_slot_base[d + 1];
  SS_CHECK_OR(s0 >= 0 && s0 <= s1 && s1 <= P.caps.slots && P.dec_tok[d] >= 0 && P.dec_tok[d] < P.total_q, &P.hdr->status,
              return);
  float m = -INFINITY;
  for (int s = s0 + lane; s < s1; s += 32) m = fmaxf(m, __ldcg(P.part_lse + static_cast<int64_t>(s) * P.Hq + h));
  m = warp_max(m);
  RowState r;
  r.acc[0] = r.acc[1] = r.acc[2] = r.acc[3] = 0.f;
  r.l = 0.f;
  r.m = m;
  if (m > -INFINITY) {
    for (int s = s0; s < s1; ++s) {
      const float ls = __ldcg(P.part_lse + static_cast<int64_t>(s) * P.Hq + h);
      if (ls == -INFINITY) continue;
      const float wgt = __expf(ls - m);
      const float4 o = __ldcg(reinterpret_cast<const float4*>(P.part_o + (static_cast<int64_t>(s) * P.Hq + h) * kHeadDim + 4 * lane));
      r.l += wgt;
      r.acc[0] += wgt * o.x; r.acc[1] += wgt * o.y; r.acc[2] += wgt * o.z; r.acc[3] += wgt * o.w;
    }
  }
  row_store_final(r, P, P.dec_tok[d], h, lane);
}

// The same merge for up to 8 rows at once (one whole warp): lane r < n_rows brings decode token `d` and q head `h` of row r.
// Three trips to memory for up to 2 partials a row (slots; log-sum-exps and values together), one more for every further
// two: a merge is nothing but latency.  Out of line (inlined it takes registers and instruction-cache space from the leaf
// kernel's page loop), with its arguments by value: through a reference to the kernel's parameters every one of them would
// be a load (5 us a call, measured).
struct MergeArgs {       // what a merge needs of Params, in registers (it is called out of line)
  const int32_t *dec_slot_base, *dec_tok;
  const float *part_o, *part_lse;
  __nv_bfloat16* out;
  float* lse;
  int32_t Hq;
#ifdef SS_CHECKED
  int64_t slots, total_q;
  int32_t* status;
#endif
};
__device__ __forceinline__ MergeArgs merge_args(const Params& P) {
  MergeArgs M{P.dec_slot_base, P.dec_tok, P.part_o, P.part_lse, P.out, P.lse, P.Hq};
#ifdef SS_CHECKED
  M.slots = P.caps.slots;
  M.total_q = P.total_q;
  M.status = &P.hdr->status;
#endif
  return M;
}
static __device__ __noinline__ void merge_rows8(const MergeArgs P, int d, int h, int n_rows, int lane) {
  int s0 = 0, ns = 0, q_row = -1;
  if (lane < n_rows) {
    s0 = __ldcg(P.dec_slot_base + d);
    ns = __ldcg(P.dec_slot_base + d + 1) - s0;
    q_row = __ldcg(P.dec_tok + d);
    SS_CHECK_OR(s0 >= 0 && ns >= 0 && s0 + ns <= P.slots && q_row >= 0 && q_row < P.total_q, P.status, { ns = 0; q_row = -1; });
  }
  const int ns_max = __reduce_max_sync(0xffffffffu, ns);
  // lane r + 8 k looks after slot 4 p + k of row r
  const int r = lane & 7, k = lane >> 3;
  const int my_s0 = __shfl_sync(0xffffffffu, s0, r), my_ns = __shfl_sync(0xffffffffu, ns, r), my_h = __shfl_sync(0xffffffffu, h, r);
  auto lse_of = [&](int p) {
    return 4 * p + k < my_ns ? __ldcg(P.part_lse + static_cast<int64_t>(my_s0 + 4 * p + k) * P.Hq + my_h) : -INFINITY;
  };
  auto value = [&](int row, int slot) {                        // (row: a constant after unrolling)
    const int rs0 = __shfl_sync(0xffffffffu, s0, row), rns = __shfl_sync(0xffffffffu, ns, row), rh = __shfl_sync(0xffffffffu, h, row);
    return slot < rns ? __ldcg(reinterpret_cast<const float4*>(P.part_o + (static_cast<int64_t>(rs0 + slot) * P.Hq + rh) * kHeadDim + 4 * lane))
                      : make_float4(0.f, 0.f, 0.f, 0.f);
  };
  float lse = lse_of(0), m = lse;
  for (int p = 1; 4 * p < ns_max; ++p) m = fmaxf(m, lse_of(p));
  float4 v[2][8];
#pragma unroll
  for (int x = 0; x < 8; ++x) { v[0][x] = value(x, 0); v[1][x] = value(x, 1); }
  m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 8));
  m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 16));
  float4 acc[8];
#pragma unroll
  for (int x = 0; x < 8; ++x) acc[x] = make_float4(0.f, 0.f, 0.f, 0.f);
  float l = 0.f, w = 0.f;
#pragma unroll 1
  for (int s = 0; s < ns_max; s += 2) {
    if ((s & 3) == 0) {
      if (s) lse = lse_of(s >> 2);
      w = lse == -INFINITY ? 0.f : __expf(lse - m);            // (m = -inf only if every one is)
      l += w;
    }
#pragma unroll
    for (int x = 0; x < 8; ++x) {
      const float w0 = __shfl_sync(0xffffffffu, w, x + 8 * (s & 3)), w1 = __shfl_sync(0xffffffffu, w, x + 8 * (s & 3) + 8);
      if (w0 != 0.f) { acc[x].x += w0 * v[0][x].x; acc[x].y += w0 * v[0][x].y; acc[x].z += w0 * v[0][x].z; acc[x].w += w0 * v[0][x].w; }
      if (w1 != 0.f) { acc[x].x += w1 * v[1][x].x; acc[x].y += w1 * v[1][x].y; acc[x].z += w1 * v[1][x].z; acc[x].w += w1 * v[1][x].w; }
    }
    if (s + 2 < ns_max) {
#pragma unroll
      for (int x = 0; x < 8; ++x) { v[0][x] = value(x, s + 2); v[1][x] = value(x, s + 3); }
    }
  }
  l += __shfl_xor_sync(0xffffffffu, l, 8);
  l += __shfl_xor_sync(0xffffffffu, l, 16);
#pragma unroll
  for (int x = 0; x < 8; ++x) {
    const int row = __shfl_sync(0xffffffffu, q_row, x), rh = __shfl_sync(0xffffffffu, h, x);
    const float sum = __shfl_sync(0xffffffffu, l, x), top = __shfl_sync(0xffffffffu, m, x);
    if (row < 0) continue;
    const float inv = sum > 0.f ? 1.f / sum : 0.f;
    const __nv_bfloat162 a = __floats2bfloat162_rn(acc[x].x * inv, acc[x].y * inv), b = __floats2bfloat162_rn(acc[x].z * inv, acc[x].w * inv);
    uint2 u;
    u.x = *reinterpret_cast<const uint32_t*>(&a);
    u.y = *reinterpret_cast<const uint32_t*>(&b);
    *reinterpret_cast<uint2*>(P.out + (static_cast<int64_t>(row) * P.Hq + rh) * kHeadDim + 4 * lane) = u;
    if (P.lse && lane == 0) P.lse[static_cast<int64_t>(row) * P.Hq + rh] = sum > 0.f ? top + __logf(sum) : -INFINITY;
  }
}

// Rows of GENERIC paths: warp `w` of `warps` takes rows w, w + warps, ... of all (query token, q head) rows.
__device__ inline void generic_rows(const Params& P, int64_t w, int64_t warps, int lane) {
  const int live = P.hdr->live_paths;
  if (live <= 0) return;
  const int64_t total_rows = P.q_offsets[live] * P.Hq;
  for (; w < total_rows; w += warps) {
    const int64_t q_row = w / P.Hq;
    const int h = static_cast<int>(w % P.Hq);
    int lo = 0, hi = live;                    // path with q_offsets[p] <= q_row < q_offsets[p+1]
    while (hi - lo > 1) {
      const int mid = (lo + hi) >> 1;
      if (P.q_offsets[mid] <= q_row) lo = mid; else hi = mid;
    }
    const int p = lo;
    if (P.path_class[p] != kClassGeneric) continue;
    const int T = P.path_q_len[p];
    const int t = static_cast<int>(q_row - P.q_offsets[p]);
    const int visible = P.path_kv_len[p] - T + t + 1;
    RowState r;
    const int64_t q_src = P.q_src_offsets ? P.q_src_offsets[p] + t : q_row;
    row_init(r, P.q + (q_src * P.Hq + h) * kHeadDim, lane);
    if (visible > 0) row_visit_chain(r, P, P.path_leaf_node[p], h / P.G, 0, visible, lane);
    row_store_final(r, P, q_row, h, lane);
  }
}

}  // namespace attn
}  // namespace ss
