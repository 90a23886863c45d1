// ss_candidate_step_host: one pass of the whole candidate-path hot path for a caller whose per-step data lives in
// HOST memory.  It only strings together what the library already exports - asynchronous copies of the step's
// inputs into a caller-owned device arena, ss_candidate_step, asynchronous copies of every result back - all on the caller's stream, without a host
// synchronisation, so that a caller that alternates between a few arenas and streams overlaps one step's copies
// with another step's kernels.
//
// Rows nobody reads need not come back over the bus: a duplicate candidate gets no forward pass (paper, Section
// "Computation Deduplication"), so it has no output of its own.  With SS_STEP_COMPACT_TRANSFERS, and out / lse
// page-locked and mapped into the device's address space, only the live rows of out / lse - the first
// u_q_offsets[num_unique], a number only the device knows - are returned, by a small kernel that writes them
// straight into the host buffers.  The query rows still go in whole, with one cudaMemcpyAsync: fetching only the
// unique paths' rows was measured and is not kept - as one copy per run of unique paths (after a host wait for the
// deduplication) the ~2700 copies of a C5 step cost more than the 20 % of the bytes they save (each costs about as
// much bus time as the 512 KB gap it skips, and the wait keeps the steps from overlapping: 135 ms per step against
// 98 ms), and as a kernel reading mapped host memory the two directions together reach only 56-80 GB/s against the
// 96 GB/s of two copy engines.
//
// Small arrays (a copy of a few KB costs its place in the stream, 2 to 4 us, whatever its size; a decode step has 8 in and
// 9 out) go through one kernel per direction that reads or writes the mapped host memory, if it is page-locked; arrays
// above kSmallBytes keep their copy engine.  Measured, a step of 1024 decode paths: 330 -> 278 us; with the query rows on a stream of
// their own, the arrays moved side by side and the rows written by the attention kernels 280 -> 214.  Arrays that do not start on 16
// bytes are read and written in the whole words of host memory that they cover, with single bytes at their two ends (all arrays an
// element off: 8 paths a byte a thread 81 us a step, 16 bytes a thread one by one 73, so 52; 1024 335, 312, 248; 4096 943, 915, 802).
#include "step.cuh"

namespace ss {
namespace host_step {

constexpr size_t kSmallBytes = 64 << 10;      // three sets in flight, 4096 decode paths: 4 KB 471 us a step, 16 KB 420, 64 KB 350, 256 KB
                                              // 350; one at a time, 1024 paths: 227, 207, 206, 208; 16384: 2341, 2332, 2297, 2282
constexpr int kMaxSegments = 12;

// Arrays to move, as one sequence of units of 16 bytes (the first and the last of an array may be shorter): a thread has a unit,
// whichever array it is of, so that a trip over the bus serves all of them (array after array, eight of them took 17 us of a
// decode step).  An array's units start on 16 bytes of HOST memory, behind a first one of `head` bytes if it does not: what goes
// over the bus is whole 16-byte words side by side, and the device side, which may lie off them then, is in the L2.
struct Segments {
  const char* src[kMaxSegments];
  char* dst[kMaxSegments];
  unsigned int bytes[kMaxSegments], head[kMaxSegments], first[kMaxSegments];   // first: unit
  unsigned int units;
  int count;
};

// The device's address of `bytes` of host memory, or null if they are not page-locked, to the last byte (an array may run past the
// end of a registered range: a copy then reports it, a kernel would fault.  Pages are locked whole, so one that lies in a page
// is only asked for once; a lookup costs the host 0.1 us).
static char* mapped(const void* host, size_t bytes) {
  if (!host || bytes == 0) return nullptr;
  char* at = static_cast<char*>(const_cast<void*>(host));
  char* end = at + bytes - 1;
  void *first = nullptr, *last = nullptr;
  const bool one_page = ((reinterpret_cast<uintptr_t>(at) ^ reinterpret_cast<uintptr_t>(end)) >> 12) == 0;
  if (cudaHostGetDevicePointer(&first, at, 0) != cudaSuccess || (!one_page && cudaHostGetDevicePointer(&last, end, 0) != cudaSuccess)) {
    (void)cudaGetLastError();
    return nullptr;
  }
  return one_page || static_cast<char*>(last) - static_cast<char*>(first) == end - at ? static_cast<char*>(first) : nullptr;
}

// Up to 16 bytes that start anywhere.  (Not inlined: a kernel that runs once and for 2 us is bound by its instruction fetches too;
// with these in line a step of 8 paths takes 3 us more.)
__device__ __noinline__ uint4 load_bytes(const char* p, unsigned int n) {
  uint32_t w[4] = {0, 0, 0, 0};
  if (n == 16 && (reinterpret_cast<uintptr_t>(p) & 3) == 0) {
#pragma unroll
    for (int x = 0; x < 4; ++x) w[x] = reinterpret_cast<const uint32_t*>(p)[x];
  } else {
#pragma unroll
    for (int x = 0; x < 16; ++x)
      if (x < n) w[x >> 2] |= static_cast<uint32_t>(static_cast<unsigned char>(p[x])) << (8 * (x & 3));
  }
  return make_uint4(w[0], w[1], w[2], w[3]);
}
__device__ __noinline__ void store_bytes(char* p, uint4 v, unsigned int n) {
  const uint32_t w[4] = {v.x, v.y, v.z, v.w};
  if (n == 16 && (reinterpret_cast<uintptr_t>(p) & 3) == 0) {
#pragma unroll
    for (int x = 0; x < 4; ++x) reinterpret_cast<uint32_t*>(p)[x] = w[x];
  } else {
#pragma unroll
    for (int x = 0; x < 16; ++x)
      if (x < n) p[x] = static_cast<char>(w[x >> 2] >> (8 * (x & 3)));
  }
}

__device__ __forceinline__ void move_segments(const Segments& S, int block, int n_blocks) {
  constexpr int kAhead = 4;
  const unsigned int step = n_blocks * blockDim.x;
  for (unsigned int u0 = block * blockDim.x + threadIdx.x; u0 < S.units; u0 += kAhead * step) {
    uint4 v[kAhead];
    char* dst[kAhead];
    unsigned int n[kAhead];
#pragma unroll
    for (int a = 0; a < kAhead; ++a) {
      const unsigned int u = u0 + a * step;
      n[a] = 0;
      dst[a] = nullptr;
      v[a] = make_uint4(0, 0, 0, 0);
      if (u >= S.units || u < u0) continue;
      int i = 0;
      while (i + 1 < S.count && S.first[i + 1] <= u) ++i;
      const unsigned int k = u - S.first[i], head = S.head[i], at = head == 0 ? 16 * k : k == 0 ? 0 : head + 16 * (k - 1);
      const char* src = S.src[i] + at;
      dst[a] = S.dst[i] + at;
      n[a] = min(head != 0 && k == 0 ? head : 16u, S.bytes[i] - at);
      if (n[a] == 16 && (reinterpret_cast<uintptr_t>(src) & 15) == 0)
        v[a] = *reinterpret_cast<const uint4*>(src);
      else
        v[a] = load_bytes(src, n[a]);
    }
#pragma unroll
    for (int a = 0; a < kAhead; ++a) {
      if (n[a] == 16 && (reinterpret_cast<uintptr_t>(dst[a]) & 15) == 0)
        *reinterpret_cast<uint4*>(dst[a]) = v[a];
      else if (n[a] > 0)
        store_bytes(dst[a], v[a], n[a]);
    }
  }
}

constexpr int kCopyBlocks = 8;       // persistent blocks of the copy kernel (8 reach 52 GB/s on the measured system)
constexpr int kCopyThreads = 512;

// The small results, and with `out_host` the live rows of out / lse, device -> (mapped) host: rows [0, u_q_offsets[U]) of the
// compact device buffers.
__global__ void __launch_bounds__(kCopyThreads)
rows_to_host_kernel(const uint4* __restrict__ out_dev, uint4* __restrict__ out_host, const uint4* __restrict__ lse_dev,
                    uint4* __restrict__ lse_host, const int32_t* __restrict__ num_unique, int32_t n_paths,
                    const int64_t* __restrict__ u_q_offsets, int64_t out_row_chunks, int64_t lse_row_bytes,
                    const __grid_constant__ Segments small) {
  ss::grid_dependency_enter();
  move_segments(small, blockIdx.x, gridDim.x);
  if (!out_host) return;
  int live = *num_unique;
  live = live < 0 ? 0 : (live > n_paths ? n_paths : live);
  const int64_t rows = u_q_offsets[live];
  const int64_t tid = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  const int64_t nt = static_cast<int64_t>(gridDim.x) * blockDim.x;
  const int64_t n_out = rows * out_row_chunks;
  for (int64_t c0 = tid; c0 < n_out; c0 += 8 * nt) {
    uint4 v[8];
#pragma unroll
    for (int x = 0; x < 8; ++x)
      if (c0 + x * nt < n_out) v[x] = out_dev[c0 + x * nt];
#pragma unroll
    for (int x = 0; x < 8; ++x)
      if (c0 + x * nt < n_out) out_host[c0 + x * nt] = v[x];
  }
  if (lse_host) {
    const int64_t n_bytes = rows * lse_row_bytes, n_lse = n_bytes / 16;
    for (int64_t c = tid; c < n_lse; c += nt) lse_host[c] = lse_dev[c];
    const float* tail_src = reinterpret_cast<const float*>(lse_dev + n_lse);       // (< 16 bytes)
    float* tail_dst = reinterpret_cast<float*>(lse_host + n_lse);
    if (tid < (n_bytes - n_lse * 16) / 4) tail_dst[tid] = tail_src[tid];
  }
}

// The small input arrays, a block's worth of threads for each 8 KB.
__global__ void __launch_bounds__(kCopyThreads) small_inputs_kernel(const __grid_constant__ Segments small) {
  ss::grid_dependency_enter();
  move_segments(small, blockIdx.x, gridDim.x);
}

struct Arena {                       // device-side layout of one step
  // staged inputs
  int32_t* tok_ids; int64_t* tok_offsets; int64_t* ctx_key; int32_t* slot_in;
  int32_t* path_leaf_node; int32_t* path_q_len; int64_t* q_offsets; void* q;
  float* scores; int32_t* seg_offsets;
  // results
  int32_t* canon; int32_t* path_to_unique; int32_t* unique_paths; int32_t* multiplicity; int32_t* slot_out;
  int32_t* num_unique;
  int32_t* u_leaf; int32_t* u_q_len; int64_t* u_q_offsets; int64_t* u_q_src;
  void* out; float* lse; int32_t* survivors; uint8_t* keep;
  // workspaces of the three calls
  void* dedup_ws; size_t dedup_ws_bytes;
  void* attn_ws; size_t attn_ws_bytes;
  void* topk_ws; size_t topk_ws_bytes;
  size_t total;
};

// The copy of the query rows on a stream of its own: behind what `st` holds when it starts (the arena's last user), in front of
// what waits for `ready`.  However the call ends, `st` waits for it.
struct QueryCopy {
  cudaStream_t st, other;
  cudaEvent_t ready = nullptr;
  bool start(void* dst, const void* src, size_t bytes) {
    cudaEvent_t begin = nullptr;
    bool ok = cudaEventCreateWithFlags(&begin, cudaEventDisableTiming) == cudaSuccess &&
              cudaEventCreateWithFlags(&ready, cudaEventDisableTiming) == cudaSuccess && cudaEventRecord(begin, st) == cudaSuccess &&
              cudaStreamWaitEvent(other, begin, 0) == cudaSuccess;
    if (ok) {
      const bool copied = cudaMemcpyAsync(dst, src, bytes, cudaMemcpyHostToDevice, other) == cudaSuccess;
      ok = cudaEventRecord(ready, other) == cudaSuccess && copied;
    }
    if (begin) cudaEventDestroy(begin);                        // (an event in use goes when it is through)
    if (!ok) (void)cudaGetLastError();
    return ok;
  }
  ~QueryCopy() {
    if (!ready) return;
    if (cudaStreamWaitEvent(st, ready, 0) != cudaSuccess) (void)cudaGetLastError();
    cudaEventDestroy(ready);
  }
};

static size_t at_least_one(int64_t n) { return static_cast<size_t>(n > 0 ? n : 1); }

// The attention descriptor of this step: the caller's resident fields + the staged per-path arrays.
static ss_attn_desc_t step_desc(const ss_host_step_t& s, const Arena& a) {
  ss_attn_desc_t d = *s.attn;
  d.num_paths = s.n_paths;
  d.num_paths_dev = a.num_unique;
  d.path_leaf_node = a.u_leaf;
  d.path_q_len = a.u_q_len;
  d.q_offsets = a.u_q_offsets;
  d.total_q = s.total_q;
  d.q_src_offsets = a.u_q_src;
  d.q_src_rows = s.total_q;
  d.q = a.q;
  d.out = a.out;
  d.lse = a.lse;
  return d;
}

static int32_t carve(const ss_host_step_t& s, void* base, Arena* a) {
  Carver c(base);
  const size_t N = at_least_one(s.n_paths), P = at_least_one(s.n_segments);
  const size_t row = static_cast<size_t>(s.attn->num_q_heads) * static_cast<size_t>(s.attn->head_dim);
  a->tok_ids = c.take<int32_t>(at_least_one(s.total_tok));
  a->tok_offsets = c.take<int64_t>(N + 1);
  a->ctx_key = c.take<int64_t>(N);
  a->slot_in = c.take<int32_t>(N);
  a->path_leaf_node = c.take<int32_t>(N);
  a->path_q_len = c.take<int32_t>(N);
  a->q_offsets = c.take<int64_t>(N + 1);
  a->q = c.take<__nv_bfloat16>(at_least_one(s.total_q) * row);
  a->scores = c.take<float>(N);
  a->seg_offsets = c.take<int32_t>(P + 1);
  a->canon = c.take<int32_t>(N);
  a->path_to_unique = c.take<int32_t>(N);
  a->unique_paths = c.take<int32_t>(N);
  a->multiplicity = c.take<int32_t>(N);
  a->slot_out = c.take<int32_t>(N);
  a->num_unique = c.take<int32_t>(1);
  a->u_leaf = c.take<int32_t>(N);
  a->u_q_len = c.take<int32_t>(N);
  a->u_q_offsets = c.take<int64_t>(N + 1);
  a->u_q_src = c.take<int64_t>(N);
  a->out = c.take<__nv_bfloat16>(at_least_one(s.total_q) * row);
  a->lse = c.take<float>(at_least_one(s.total_q) * static_cast<size_t>(s.attn->num_q_heads));
  a->survivors = c.take<int32_t>(P * static_cast<size_t>(s.top_k));
  a->keep = c.take<uint8_t>(N);
  int32_t rc = ss_dedup_workspace_bytes(s.n_paths, &a->dedup_ws_bytes);
  if (rc != SS_OK) return rc;
  a->dedup_ws = c.take<char>(a->dedup_ws_bytes);
  const ss_attn_desc_t d = step_desc(s, *a);
  rc = ss_tree_attention_workspace_bytes(&d, &a->attn_ws_bytes);
  if (rc != SS_OK) return rc;
  a->attn_ws = c.take<char>(a->attn_ws_bytes);
  rc = ss_topk_workspace_bytes(s.n_paths, &a->topk_ws_bytes);
  if (rc != SS_OK) return rc;
  a->topk_ws = c.take<char>(a->topk_ws_bytes);
  a->total = c.off;
  return SS_OK;
}

static int32_t check(const ss_host_step_t* s) {
  if (!s || s->struct_size != sizeof(ss_host_step_t) || !s->attn) return SS_ERR_INVALID_ARG;
  if (s->attn->struct_size != sizeof(ss_attn_desc_t)) return SS_ERR_INVALID_ARG;
  if (s->flags & ~SS_STEP_COMPACT_TRANSFERS) return SS_ERR_INVALID_ARG;
  if (s->n_paths < 0 || s->n_segments < 0 || s->top_k < 1 || s->total_tok < 0 || s->total_q < 0)
    return SS_ERR_INVALID_ARG;
  if (s->attn->num_q_heads < 1 || s->attn->head_dim < 1) return SS_ERR_INVALID_ARG;
  return SS_OK;
}

}  // namespace host_step
}  // namespace ss

extern "C" int32_t ss_candidate_step_host_arena_bytes(const ss_host_step_t* step, size_t* out_bytes) {
  using namespace ss::host_step;
  if (!out_bytes) return SS_ERR_INVALID_ARG;
  int32_t rc = check(step);
  if (rc != SS_OK) return rc;
  Arena a;
  rc = carve(*step, nullptr, &a);        // offsets only: nothing is dereferenced
  if (rc != SS_OK) return rc;
  *out_bytes = a.total;
  return SS_OK;
}

extern "C" int32_t ss_candidate_step_host(const ss_host_step_t* step, void* device_arena, size_t arena_bytes,
                                          void* stream) {
  return ss_candidate_step_host_2(step, device_arena, arena_bytes, stream, nullptr);
}

extern "C" int32_t ss_candidate_step_host_2(const ss_host_step_t* step, void* device_arena, size_t arena_bytes,
                                            void* stream, void* copy_stream) {
  using namespace ss;
  using namespace ss::host_step;
  int32_t rc = check(step);
  if (rc != SS_OK) return rc;
  const ss_host_step_t& s = *step;
  if (!device_arena || reinterpret_cast<uintptr_t>(device_arena) % kAlign) return SS_ERR_INVALID_ARG;
  if (!s.tok_offsets || !s.path_leaf_node || !s.path_q_len || !s.q_offsets || !s.seg_offsets || !s.canon ||
      !s.path_to_unique || !s.unique_paths || !s.multiplicity || !s.num_unique || !s.u_q_offsets || !s.survivors ||
      !s.device_status)
    return SS_ERR_INVALID_ARG;
  if ((s.slot_in == nullptr) != (s.slot_out == nullptr)) return SS_ERR_INVALID_ARG;
  if (s.n_paths > 0 && (!s.scores || !s.keep)) return SS_ERR_INVALID_ARG;
  if (s.total_tok > 0 && !s.tok_ids) return SS_ERR_INVALID_ARG;
  if (s.total_q > 0 && (!s.q || !s.out)) return SS_ERR_INVALID_ARG;
  Arena a;
  rc = carve(s, device_arena, &a);
  if (rc != SS_OK) return rc;
  if (arena_bytes < a.total) return SS_ERR_WORKSPACE_TOO_SMALL;
  cudaStream_t st = as_stream(stream);
  const size_t N = static_cast<size_t>(s.n_paths), P = static_cast<size_t>(s.n_segments);
  const size_t row = static_cast<size_t>(s.attn->num_q_heads) * static_cast<size_t>(s.attn->head_dim);
  const size_t q_bytes = static_cast<size_t>(s.total_q) * row * sizeof(__nv_bfloat16);
  const size_t lse_bytes = static_cast<size_t>(s.total_q) * static_cast<size_t>(s.attn->num_q_heads) * sizeof(float);

  // ---- host -> device: the step's candidates, queries and scores ------------------------------------------------
  Segments in{}, res{};
  // puts an array on the list if it is small and mapped; else copies it
  auto move = [&](Segments& list, void* dst, const void* src, size_t bytes, bool to_host) -> bool {
    if (bytes == 0) return true;
    char* map = bytes <= kSmallBytes && list.count < kMaxSegments ? mapped(to_host ? dst : src, bytes) : nullptr;
    if (!map) {
      if (cudaMemcpyAsync(dst, src, bytes, to_host ? cudaMemcpyDeviceToHost : cudaMemcpyHostToDevice, st) == cudaSuccess) return true;
      (void)cudaGetLastError();
      return false;
    }
    list.src[list.count] = to_host ? static_cast<const char*>(src) : map;
    list.dst[list.count] = to_host ? map : static_cast<char*>(dst);
    const size_t head = (0 - reinterpret_cast<uintptr_t>(map)) & 15;   // (bytes in front of the first whole word)
    list.head[list.count] = static_cast<unsigned int>(head);
    list.first[list.count] = list.units;
    list.units += static_cast<unsigned int>((head ? 1 : 0) + (bytes > head ? (bytes - head + 15) / 16 : 0));
    list.bytes[list.count++] = static_cast<unsigned int>(bytes);
    return true;
  };
  const bool apart = copy_stream && as_stream(copy_stream) != st && q_bytes > kSmallBytes;   // the query rows on their own stream
  bool ok = move(in, a.tok_ids, s.tok_ids, static_cast<size_t>(s.total_tok) * 4, false) &&
            move(in, a.tok_offsets, s.tok_offsets, (N + 1) * 8, false) &&
            (!s.ctx_key || move(in, a.ctx_key, s.ctx_key, N * 8, false)) &&
            (!s.slot_in || move(in, a.slot_in, s.slot_in, N * 4, false)) &&
            move(in, a.path_leaf_node, s.path_leaf_node, N * 4, false) && move(in, a.path_q_len, s.path_q_len, N * 4, false) &&
            move(in, a.q_offsets, s.q_offsets, (N + 1) * 8, false) && (apart || move(in, a.q, s.q, q_bytes, false)) &&
            move(in, a.scores, s.scores, N * 4, false) && move(in, a.seg_offsets, s.seg_offsets, (P + 1) * 4, false);
  if (!ok) return SS_ERR_CUDA;
  // compact return: needs out / lse mapped (the kernel writes them, 16 bytes at a time) and whole 16-byte chunks per row
  char *out_map = nullptr, *lse_map = nullptr;
  bool compact = (s.flags & SS_STEP_COMPACT_TRANSFERS) != 0 && s.total_q > 0 && s.n_paths > 0 &&
                 row * sizeof(__nv_bfloat16) % 16 == 0;
  if (compact) {
    out_map = mapped(s.out, q_bytes);
    if (s.lse) lse_map = mapped(s.lse, lse_bytes);
    compact = out_map && (!s.lse || lse_map) && ((reinterpret_cast<uintptr_t>(out_map) | reinterpret_cast<uintptr_t>(lse_map)) & 15) == 0;
  }
  if (in.count > 0) {
    const int blocks = static_cast<int>((in.units + kCopyThreads - 1) / kCopyThreads);
    SS_LAUNCH(small_inputs_kernel, blocks < kCopyBlocks ? blocks : kCopyBlocks, kCopyThreads, 0, st, in);
  }

  // The query rows, which nothing in front of the attention kernels reads: with a second stream they are on their way (62 us for
  // 1024 paths of 12 heads) while the candidates are deduplicated and the attention is planned.  (Behind the small arrays, which the
  // deduplication waits for: side by side their kernel took 27 us instead of 8.)
  QueryCopy queries{st, as_stream(copy_stream)};
  if (apart && !queries.start(a.q, s.q, q_bytes)) return SS_ERR_CUDA;

  // ---- the path ---------------------------------------------------------------------------------------------------
  ss_attn_desc_t d = step_desc(s, a);
  // Decode rows (one a path) can be written to the caller's memory by the attention kernels themselves, as the leaves are done:
  // their 16-byte stores keep the bus as busy as a copy kernel behind them does.
  const bool direct = compact && s.total_q == s.n_paths && reinterpret_cast<uintptr_t>(out_map) % 32 == 0;
  if (direct) d.out = out_map;
  if (compact && !direct && d.max_sms == 0) {
    // the copy kernel of the step before this one (another stream) runs for as long as the bus takes and needs SMs
    // that this step's persistent attention blocks do not hold
    int dev = 0, n_sm = 0;
    if (cudaGetDevice(&dev) == cudaSuccess && cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess &&
        n_sm > 4 * kCopyBlocks)
      d.max_sms = n_sm - 2 * kCopyBlocks;
    else
      (void)cudaGetLastError();
  }
  ss_device_step_t p{};
  p.struct_size = sizeof p;
  p.dedup_flags = s.dedup_flags;
  p.attn = &d;
  p.n_paths = s.n_paths; p.n_segments = s.n_segments; p.top_k = s.top_k;
  p.dedup_workspace_bytes = a.dedup_ws_bytes; p.attn_workspace_bytes = a.attn_ws_bytes; p.topk_workspace_bytes = a.topk_ws_bytes;
  p.tok_ids = a.tok_ids; p.tok_offsets = a.tok_offsets; p.ctx_key = s.ctx_key ? a.ctx_key : nullptr;
  p.slot_in = s.slot_in ? a.slot_in : nullptr;
  p.path_leaf_node = a.path_leaf_node; p.path_q_len = a.path_q_len; p.q_offsets = a.q_offsets;
  p.scores = a.scores; p.seg_offsets = a.seg_offsets;
  p.canon = a.canon; p.path_to_unique = a.path_to_unique; p.unique_paths = a.unique_paths; p.multiplicity = a.multiplicity;
  p.slot_out = s.slot_in ? a.slot_out : nullptr; p.num_unique = a.num_unique;
  p.u_leaf = a.u_leaf; p.u_q_len = a.u_q_len; p.u_q_offsets = a.u_q_offsets; p.u_q_src = a.u_q_src;
  p.survivors = a.survivors; p.keep = a.keep;
  p.dedup_workspace = a.dedup_ws; p.attn_workspace = a.attn_ws; p.topk_workspace = a.topk_ws;
  rc = candidate_step(p, stream, queries.ready, direct);
  if (rc != SS_OK) return rc;

  // ---- device -> host: every result ------------------------------------------------------------------------------------
  if (!compact)
    ok = move(res, s.out, a.out, q_bytes, true) &&
         (!s.lse || move(res, s.lse, a.lse, lse_bytes, true));
  ok = ok && move(res, s.canon, a.canon, N * 4, true) && move(res, s.path_to_unique, a.path_to_unique, N * 4, true) &&
       move(res, s.unique_paths, a.unique_paths, N * 4, true) && move(res, s.multiplicity, a.multiplicity, N * 4, true) &&
       (!s.slot_out || move(res, s.slot_out, a.slot_out, N * 4, true)) && move(res, s.num_unique, a.num_unique, 4, true) &&
       move(res, s.u_q_offsets, a.u_q_offsets, (N + 1) * 8, true) &&
       move(res, s.survivors, a.survivors, P * static_cast<size_t>(s.top_k) * 4, true) && move(res, s.keep, a.keep, N, true) &&
       move(res, s.device_status, a.attn_ws, sizeof(int32_t), true);   // first word of the attention workspace
  if (!ok) return SS_ERR_CUDA;
  if (compact || res.count > 0)
    SS_LAUNCH(rows_to_host_kernel, kCopyBlocks, kCopyThreads, 0, st, static_cast<const uint4*>(a.out),
              reinterpret_cast<uint4*>(compact ? out_map : nullptr), reinterpret_cast<const uint4*>(a.lse),
              reinterpret_cast<uint4*>(lse_map), static_cast<const int32_t*>(a.num_unique), s.n_paths,
              static_cast<const int64_t*>(a.u_q_offsets), direct ? 0 : static_cast<int64_t>(row * sizeof(__nv_bfloat16) / 16),
              static_cast<int64_t>(s.attn->num_q_heads) * 4, res);
  return SS_OK;
}
