// ss_branch_sample: the sampling half of on-demand branching (paper, Section "Computation Deduplication"): a
// sequence with potential size n draws n next tokens as independent trials from ONE logits row; equal draws are
// grouped afterwards with ss_dedup_paths on (sequence, token) pairs.
//
// The token decision is taken in fp64 (so that it agrees with a plain fp64 CPU evaluation except for draws within
// ~1e-15 of a boundary), one exponential per logit.  A row is split over the 16 warps of a block, or of a CLUSTER of
// 2, 4 or 8 blocks when there are too few rows to give every SM one: each warp has one contiguous slice, and the slice sums
// meet in (distributed) shared memory.  Nothing is read twice but the 512 tokens around each draw.
//   1. every warp sums 2^(logit_v * c), c = log2(e) / temperature, over its slice in segments of 512 tokens and keeps
//      the running sum at every segment's end (shared memory)
//   2. the slice sums are written to every block of the cluster
//   3. each of the row's warps takes a share of its draws: it finds the slice that holds u * Z from the slice sums, the
//      segment from the running sums of the slice's owner, evaluates the segment again with a warp scan, and writes the
//      token
// A block that handles several rows takes step 1 of the next row before step 3 of the current one, between the two halves
// of a split barrier, so that neither the barrier nor a draw is waited for; the warps that draw change from row to row.
// There is no pass for the maximum: fp64 holds 2^(logit * c) itself for rows whose largest exponent lies in
// [kLowTop, kHighTop], which every ordinary row does; a row outside (or a temperature outside [1e-3, 1e6]) is summed again
// relative to its maximum, and its draws are taken by the warps in whose slices they fall.
//
// The exponential (after Tang, "Table-driven implementation of the exponential function in IEEE floating-point
// arithmetic", ACM TOMS 15, 1989): K = the integer nearest to 128 * x from ONE fp32 FMA (it only has to be near), r =
// 128 * x - K exactly by one fp64 FMA, 2^(K/128) from a table of 128 entries and an integer addition to the exponent,
// 2^(r/128) by a polynomial of degree 4 (interpolated at Chebyshev nodes; relative error below 1.6e-16 for |r| <= 0.505, 1.8e-16 for
// 0.508, which the fp32 rounding of 128 * c allows at the largest exponents).
// 8 fp64 instructions with the summation; the table is copied 16 times so that every lane reads its own bank pair.
// Bound: issue slots.  An fp64 instruction holds two, so 32 logits take ~30 clocks of a sub-partition, 120 us for
// 922 x 151936 logits (the loop alone, measured; 4 bytes a logit from HBM would take 85).  Measured, the call: 922 rows
// 582 -> 182 us, 16 rows 91 -> 12.4 us, against one block of 1024 threads per row with a pass for the maximum, CUDA's exp
// and a block-wide scan for every 4096 tokens.
#include <cooperative_groups.h>

#include "common.cuh"

namespace ss {
namespace sample {

namespace cg = cooperative_groups;

constexpr int kThreads = 512;                                 // one block per SM (128 registers a thread)
constexpr int kWarps = kThreads / 32;
constexpr int kSeg = 512;                                     // tokens per segment: 16 per lane, 4 x 128 bits
constexpr int kMaxSegs = 32;                                  // per slice
constexpr int kMaxVocab = 2097152;
constexpr int kTable = 128;
constexpr int kLater = -1;                                    // not a token
constexpr float kLowTop = -200.f, kHighTop = 900.f;           // exponent range of a row's largest term
constexpr float kLowest = -1020.f;                            // smaller exponents count as this one (2^-820 of the sum)
constexpr double kTiny = 1e-300;                              // above 2^-1020: what a masked token counts for

struct Args {
  const float* logits;
  const int64_t* draw_offsets;
  const float* uniforms;
  int32_t* tokens_out;
  int64_t* seq_out;
  int n_seq, row0, vocab;
  int slice;                   // tokens per warp, a multiple of kSeg / 2
  int many;                    // draws of a row from which its segments are gone through instead
  double inv_temperature;
  double ck;                   // kTable * log2(e) / temperature
  float ckf, lowest;           // lowest: the logit whose exponent is kLowest
  double lowest_below;         // the same for l - dm
  bool fast;                   // the temperature allows sums that are not relative to the row's maximum
};

template <int CL>
struct Sums {                          // of one row
  double seg_end[kWarps][kMaxSegs];    // own slices: sum up to the end of each segment
  double slice_sum[CL * kWarps];       // the whole row's, written by the cluster's blocks
  float slice_max[CL * kWarps];
};
template <int CL>
struct Shared {
  double table[kTable * 16];
  Sums<CL> sums[3];                    // rows in turn (a warp may be two rows ahead of one that reads its running sums)
  int queue[kWarps][64];               // see row_below
};

// 2^(K / 128) * 2^(r / 128) (see the head of the file); `bits`: K in the low bits, nothing in the ones above that the shift keeps;
// `bank` = table + (lane & 15)
__device__ __forceinline__ double exp2_parts(int bits, double r, const double* bank) {
  constexpr double a1 = 0.005415212348124257, a2 = 1.466226238764014e-05, a3 = 2.6466431340771855e-08,
                   a4 = 3.5830331985890313e-11;
  const double t0 = bank[(bits & (kTable - 1)) * 16];
  // K / 128 into the exponent field: the table has K % 128 taken off again
  const double t = __hiloint2double(__double2hiint(t0) + (bits << 13), __double2loint(t0));
  double q = fma(a4, r, a3);
  q = fma(q, r, a2);
  q = fma(q, r, a1);
  return fma(t * r, q, t);
}
// 2^(l * c) for -1021 < l * c < 1021
__device__ __forceinline__ double exp2_table(float l, const Args& A, const double* bank) {
  constexpr float kRound = 12582912.f;                        // 1.5 * 2^23: the sum's low bits are the nearest integer
  const int bits = __float_as_int(fmaf(l, A.ckf, kRound));    // 0x4b400000 + K
  const double K = __hiloint2double(0x43300000, bits) - (4503599627370496.0 + 1262485504.0);   // 2^52 + bits - (2^52 + 0x4b400000)
  return exp2_parts(bits, fma(static_cast<double>(l), A.ck, -K), bank);
}
// 2^((l - dm) * c) for l <= dm at any temperature: K from an fp64 sum.
__device__ __forceinline__ double exp2_below(float l, double dm, const Args& A, const double* bank) {
  constexpr double kRound = 6755399441055744.0;               // 1.5 * 2^52
  double d = static_cast<double>(l) - dm;
  d = d < A.lowest_below ? A.lowest_below : d;                // (a NaN stays one)
  const double k = fma(d, A.ck, kRound);
  return exp2_parts(__double2loint(k), fma(d, A.ck, -(k - kRound)), bank);
}
// The term relative to the row's maximum, exactly 0 where fp64 has nothing smaller (the table gives 2^-1020 at least, also for
// masked tokens and past the end).
__device__ __noinline__ double term_exact(float l, double dmax, double inv_temperature) {
  return exp((static_cast<double>(l) - dmax) * inv_temperature);
}

// 8 logits of a lane, half of its share of a segment: tokens base + 128 j + 4 lane + x for j = 0, 1; -inf past the end.
// VEC: rows start on 16 bytes and are whole 16-byte units.
template <bool VEC>
__device__ __forceinline__ void load_half(const float* __restrict__ row, int base, int vocab, int lane, float (&l)[8]) {
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    const int v = base + 128 * j + 4 * lane;
    if (VEC) {
      const float4 f = v < vocab ? __ldg(reinterpret_cast<const float4*>(row + v))
                                 : make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
      l[4 * j] = f.x; l[4 * j + 1] = f.y; l[4 * j + 2] = f.z; l[4 * j + 3] = f.w;
    } else {
#pragma unroll
      for (int x = 0; x < 4; ++x) l[4 * j + x] = v + x < vocab ? __ldg(row + v + x) : -INFINITY;
    }
  }
}

__device__ __forceinline__ double warp_sum_d(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Sum of the warp's slice of n_half half segments, the first of which is in `a`; `mx`: the largest logit of the lane.
template <bool VEC>
__device__ __forceinline__ double slice_sums(const float* __restrict__ row, const Args& A, const double* bank,
                                             double* seg_end, int v0, int n_half, int lane, float (&a)[8], float& mx) {
  double end = 0.0;
  mx = -INFINITY;
  float b[8];                                                  // one half in flight while the other is summed
  auto add = [&](float (&l)[8], double& s0, double& s1) {
    float mn = l[0];
#pragma unroll
    for (int x = 0; x < 8; ++x) { mx = fmaxf(mx, l[x]); mn = fminf(mn, l[x]); }
    if (__any_sync(0xffffffffu, !(mn >= A.lowest))) {          // masked tokens, or past the end (a NaN stays one)
#pragma unroll
      for (int x = 0; x < 8; ++x) asm("max.NaN.f32 %0, %1, %2;" : "=f"(l[x]) : "f"(l[x]), "f"(A.lowest));
    }
#pragma unroll
    for (int x = 0; x < 8; x += 2) {
      s0 += exp2_table(l[x], A, bank);
      s1 += exp2_table(l[x + 1], A, bank);
    }
  };
#pragma unroll 1
  for (int h = 0; h < n_half; h += 2) {
    double s0 = 0.0, s1 = 0.0;
    const bool second = h + 1 < n_half;
    if (second) load_half<VEC>(row, v0 + (h + 1) * (kSeg / 2), A.vocab, lane, b);
    add(a, s0, s1);
    if (second) {
      if (h + 2 < n_half) load_half<VEC>(row, v0 + (h + 2) * (kSeg / 2), A.vocab, lane, a);
      add(b, s0, s1);
    }
    end += warp_sum_d(s0 + s1);
    if (lane == 0) seg_end[h >> 1] = end;
  }
  return end;
}
// The same relative to the row's maximum dm.
template <bool VEC>
__device__ __forceinline__ double slice_sums_below(const float* __restrict__ row, const Args& A, const double* bank,
                                                   double* seg_end, int v0, int n_half, int lane, double dm, float& mx) {
  double end = 0.0, s0 = 0.0, s1 = 0.0;
  mx = -INFINITY;
  float next[8];
  load_half<VEC>(row, v0, A.vocab, lane, next);
#pragma unroll 1
  for (int h = 0; h < n_half; ++h) {
    float l[8];
#pragma unroll
    for (int x = 0; x < 8; ++x) l[x] = next[x];
    if (h + 1 < n_half) load_half<VEC>(row, v0 + (h + 1) * (kSeg / 2), A.vocab, lane, next);
#pragma unroll
    for (int x = 0; x < 8; x += 2) {
      mx = fmaxf(mx, fmaxf(l[x], l[x + 1]));
      s0 += exp2_below(l[x], dm, A, bank);
      s1 += exp2_below(l[x + 1], dm, A, bank);
    }
    if ((h & 1) || h + 1 == n_half) {
      end += warp_sum_d(s0 + s1);
      s0 = s1 = 0.0;
      if (lane == 0) seg_end[h >> 1] = end;
    }
  }
  return end;
}

// The slice's sum and maximum to every block of the cluster (visible there after the cluster's next barrier).
template <int CL>
__device__ __forceinline__ void publish(cg::cluster_group& cl, Sums<CL>& S, int slice, int lane, double sum, float mx) {
  if (lane < CL) {
    Sums<CL>* R = cl.map_shared_rank(&S, lane);
    R->slice_sum[slice] = sum;
    R->slice_max[slice] = mx;
  }
}
// The two halves of the cluster's barrier (a cluster of one block: of the block's).
__device__ __forceinline__ void cluster_arrive() {
  __syncwarp();
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }

// A slice's place in its row.
struct Slice {
  int v0, n_half;                                              // n_half: half segments
};
__device__ __forceinline__ Slice slice_of(const Args& A, int slice) {
  const int64_t first = static_cast<int64_t>(slice) * A.slice;
  const int v0 = static_cast<int>(first < A.vocab ? first : A.vocab);
  return Slice{v0, (min(A.slice, A.vocab - v0) + kSeg / 2 - 1) / (kSeg / 2)};
}

// A lane's terms of the segment [base, min(base + kSeg, end)) (BELOW: relative to dm), the sums of its share of each group of 128 tokens, and their
// scans over the warp.
struct Terms {
  double e[4][4], run[4], incl[4];
};
template <bool BELOW, bool VEC>
__device__ __forceinline__ void segment_terms(Terms& T, const float* __restrict__ row, const Args& A, const double* bank,
                                              double dm, int base, int end, int lane) {
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    float l[8];
    load_half<VEC>(row, base + h * (kSeg / 2), end, lane, l);
#pragma unroll
    for (int x = 0; x < 8; ++x)
      T.e[2 * h + (x >> 2)][x & 3] = BELOW ? exp2_below(l[x], dm, A, bank) : exp2_table(fmaxf(l[x], A.lowest), A, bank);
  }
#pragma unroll
  for (int j = 0; j < 4; ++j) T.incl[j] = T.run[j] = (T.e[j][0] + T.e[j][1]) + (T.e[j][2] + T.e[j][3]);
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const double y = __shfl_up_sync(0xffffffffu, T.incl[j], o);
      if (lane >= o) T.incl[j] += y;
    }
  }
}
// The token of target t, which lies in the segment at `base`; `before`: the sum in front of it.
__device__ __forceinline__ int pick(const Terms& T, const Args& A, int base, double before, double t) {
  int token = -1;                                              // if rounding leaves t above everything: the last that counts
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const uint32_t some = __ballot_sync(0xffffffffu, T.run[j] > kTiny);
    const uint32_t over = __ballot_sync(0xffffffffu, T.run[j] > kTiny && before + T.incl[j] > t);
    if (some) {
      const int f = over ? __ffs(over) - 1 : 31 - __clz(some);
      double c = before + (T.incl[j] - T.run[j]);
      int hit = -1, tail = 0;
#pragma unroll
      for (int x = 0; x < 4; ++x) {
        c += T.e[j][x];
        if (T.e[j][x] > kTiny) {
          tail = x;
          if (hit < 0 && c > t) hit = x;
        }
      }
      token = base + 128 * j + 4 * f + __shfl_sync(0xffffffffu, hit < 0 ? tail : hit, f);
      if (over) return token;
    }
    before += __shfl_sync(0xffffffffu, T.incl[j], 31);
  }
  return token < 0 ? A.vocab - 1 : token;
}

// The row's first token whose term is not 0 at all (the sums do not tell: a masked term counts as 2^-1020 in them).  It is in
// the first slice whose largest logit's is not.  A row that is masked up to its last tokens: 16 rows of 151936 18 us, 1810 with
// a pass over the whole row.
__device__ __noinline__ int first_positive(const float* __restrict__ row, const Args& A, const float* slice_max, int n_slices,
                                           double dmax, int lane) {
  for (int s0 = 0; s0 < n_slices; s0 += 32) {
    const bool some = s0 + lane < n_slices && term_exact(slice_max[s0 + lane], dmax, A.inv_temperature) > 0.0;
    const uint32_t any = __ballot_sync(0xffffffffu, some);
    if (!any) continue;
    const int64_t first = static_cast<int64_t>(s0 + __ffs(any) - 1) * A.slice;
    const int end = static_cast<int>(min(first + A.slice, static_cast<int64_t>(A.vocab)));
    for (int v = static_cast<int>(first); v < end; v += 32 * 8) {
      float l[8];
#pragma unroll
      for (int x = 0; x < 8; ++x) l[x] = v + 32 * x + lane < end ? __ldg(row + v + 32 * x + lane) : -INFINITY;
#pragma unroll
      for (int x = 0; x < 8; ++x) {
        const uint32_t pos = __ballot_sync(0xffffffffu, term_exact(l[x], dmax, A.inv_temperature) > 0.0);
        if (pos) return v + 32 * x + __ffs(pos) - 1;
      }
    }
  }
  return A.vocab - 1;
}

// Cumulative sums at the ends of the cluster's blocks (lane b < CL: block b's) and the row's total: the first lanes add up a
// block's slices, then the blocks in turn.  A slice ends at (start of its block) + (sum of the block's slices so far), so the
// ends ascend whatever the rounding.
template <int CL>
__device__ __forceinline__ void block_ends(const Sums<CL>& S, int lane, double& end_b, double& Z) {
  double in_block = 0.0;
  end_b = Z = 0.0;
  if (lane < CL)
    for (int w = 0; w < kWarps; ++w) in_block += S.slice_sum[lane * kWarps + w];
#pragma unroll
  for (int b = 0; b < CL; ++b) {
    Z += __shfl_sync(0xffffffffu, in_block, b);
    if (lane == b) end_b = Z;
  }
}

// The token of every lane's own target, or -1 where rounding leaves it to `pick`.
__device__ __forceinline__ int pick_each(const Terms& T, int base, double before, double t) {
  double in_front = before;                                    // the group of 128, then the lane of it, that holds t
  int j = 0;
#pragma unroll
  for (int x = 0; x < 3; ++x) {
    const double e = in_front + __shfl_sync(0xffffffffu, T.incl[x], 31);
    if (j == x && !(e > t)) {
      ++j;
      in_front = e;
    }
  }
  int f = 0;
#pragma unroll
  for (int step = 16; step > 0; step >>= 1) {
    double v = 0.0;
#pragma unroll
    for (int x = 0; x < 4; ++x) {
      const double y = __shfl_sync(0xffffffffu, T.incl[x], f + step - 1);
      if (j == x) v = y;
    }
    if (!(in_front + v > t)) f += step;
  }
  double c = 0.0, e[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
  for (int x = 0; x < 4; ++x) {
    const double y = in_front + (__shfl_sync(0xffffffffu, T.incl[x], f) - __shfl_sync(0xffffffffu, T.run[x], f));
    if (j == x) c = y;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const double z = __shfl_sync(0xffffffffu, T.e[x][k], f);
      if (j == x) e[k] = z;
    }
  }
  int token = -1;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    c += e[k];
    if (token < 0 && e[k] > kTiny && c > t) token = base + 128 * j + 4 * f + k;
  }
  return token;
}

// A row outside the table's range or with many draws, mx its maximum: the sums once more, relative to it, and then the draws
// that fall into this warp's slice, a segment at a time: it is evaluated once for all of them.  `queue`: 64 words of the warp's.
template <int CL, bool VEC>
__device__ __forceinline__ void row_below(const Args& A, Sums<CL>& S, int* queue, const double* bank, int64_t seq, int slice,
                                          int lane, float mx) {
  constexpr int kSlices = CL * kWarps;
  const float* row = A.logits + seq * A.vocab;
  const int64_t d0 = A.draw_offsets[seq], d1 = A.draw_offsets[seq + 1];
  const double dm = static_cast<double>(mx);                   // (if it is not finite the sum is a NaN)
  cg::cluster_group cl = cg::this_cluster();
  {
    const Slice L = slice_of(A, slice);
    float top;
    cl.sync();                                                 // (nobody reads the sums of the row before any more)
    const double sum = slice_sums_below<VEC>(row, A, bank, S.seg_end[slice % kWarps], L.v0, L.n_half, lane, dm, top);
    publish<CL>(cl, S, slice, lane, sum, warp_max(top));
    cl.sync();
  }
  double end_b, Z;
  block_ends<CL>(S, lane, end_b, Z);
  if (slice == 0) {                                            // draws that no segment holds
    for (int64_t c = d0; c < d1; c += 32) {
      const double t = c + lane < d1 ? static_cast<double>(A.uniforms[c + lane]) * Z : 1.0;
      int token = A.vocab - 1;
      if (__any_sync(0xffffffffu, t == 0.0)) {
        const int first = first_positive(row, A, S.slice_max, kSlices, dm, lane);
        if (t == 0.0) token = first;
      }
      if (c + lane < d1 && (t == 0.0 || !(t < Z))) {
        A.tokens_out[c + lane] = token;
        A.seq_out[c + lane] = seq;
      }
    }
  }
  // The slice and its segments, by the same sums as in `draws`.  A vocabulary of few slices: several warps share the draws of one.
  const int used = static_cast<int>((static_cast<int64_t>(A.vocab) + A.slice - 1) / A.slice), parts = kSlices / used;
  const int own = slice % used, part = slice / used, block = own / kWarps, warp = own % kWarps;
  if (part >= parts) return;
  const Slice L = slice_of(A, own);
  const int n_seg = (L.n_half + 1) >> 1;
  const double block_start = __shfl_sync(0xffffffffu, end_b, max(block - 1, 0)), start = block ? block_start : 0.0;
  double in_front = 0.0;
  for (int w = 0; w < warp; ++w) in_front += S.slice_sum[block * kWarps + w];
  const double before = start + in_front, slice_end = start + (in_front + S.slice_sum[own]);
  const double end_s = lane < n_seg ? cl.map_shared_rank(&S, block)->seg_end[warp][lane] : 0.0;
  const double last_end = __shfl_sync(0xffffffffu, end_s, max(n_seg - 1, 0));
  const int s_last = __ffs(__ballot_sync(0xffffffffu, lane < n_seg && end_s == last_end)) - 1;   // (-1: no segment, or a NaN)
#pragma unroll 1
  for (int s = 0; s <= s_last; ++s) {
    const double in_slice = __shfl_sync(0xffffffffu, end_s, max(s - 1, 0)), seg_end = before + __shfl_sync(0xffffffffu, end_s, s);
    const double from = s ? before + in_slice : before, to = s == s_last ? slice_end : fmin(seg_end, slice_end);
    const double low = own == 0 && s == 0 ? -INFINITY : from;
    const int base = L.v0 + s * kSeg;
    Terms T;
    bool evaluated = false;
    int waiting = 0;                                           // draws in the queue, which are looked up 32 at a time
    auto look_up = [&](int count) {
      if (!evaluated) segment_terms<true, VEC>(T, row, A, bank, dm, base, min(A.vocab, L.v0 + A.slice), lane);
      evaluated = true;
      __syncwarp();
      const int64_t d = d0 + (lane < count ? queue[lane] : queue[0]);
      const double t = static_cast<double>(__ldg(A.uniforms + d)) * Z;
      int token = pick_each(T, base, from, t);
      for (uint32_t open = __ballot_sync(0xffffffffu, token < 0); open; open &= open - 1) {
        const int i = __ffs(open) - 1;
        const int one = pick(T, A, base, from, __shfl_sync(0xffffffffu, t, i));
        if (lane == i) token = one;
      }
      if (lane < count) {
        A.tokens_out[d] = token;
        A.seq_out[d] = seq;
      }
      __syncwarp();
    };
    constexpr int kAhead = 4;
#pragma unroll 1
    for (int64_t c0 = d0 + 32 * part; c0 < d1; c0 += 32 * kAhead * parts) {
      float u[kAhead];
#pragma unroll
      for (int k = 0; k < kAhead; ++k) {
        const int64_t d = c0 + 32 * parts * k + lane;
        u[k] = d < d1 ? __ldg(A.uniforms + d) : 2.f;           // (2: above every segment)
      }
#pragma unroll
      for (int k = 0; k < kAhead; ++k) {
        const double t = static_cast<double>(u[k]) * Z;
        const bool mine = t != 0.0 && t >= low && t < to;
        const uint32_t members = __ballot_sync(0xffffffffu, mine);
        if (!members) continue;
        if (mine) queue[waiting + __popc(members & ((1u << lane) - 1u))] = static_cast<int>(c0 - d0) + 32 * parts * k + lane;
        waiting += __popc(members);
        if (waiting >= 32) {
          look_up(32);
          waiting -= 32;
          const int moved = queue[32 + lane];
          __syncwarp();
          queue[lane] = moved;
          __syncwarp();
        }
      }
    }
    if (waiting > 0) look_up(waiting);
  }
}

// This warp's share of the draws of row `seq`; `at`: which of `sums` holds the row.  True, with nothing drawn, if the row is
// outside the table's range or has many draws (the cluster agrees).
template <int CL, bool VEC>
__device__ __forceinline__ bool draws(const Args& A, Sums<CL>* sums, const double* bank, int at, int64_t seq, int slice, int lane) {
  constexpr int kSlices = CL * kWarps;
  const int64_t d0 = A.draw_offsets[seq], d1 = A.draw_offsets[seq + 1];
  const int turn = static_cast<int>((slice + seq) % kSlices);
  float mx = -INFINITY;
  for (int i = lane; i < kSlices; i += 32) mx = fmaxf(mx, sums[at].slice_max[i]);
  mx = warp_max(mx);
  const float top = mx * A.ckf * (1.f / kTable);
  if (!(A.fast && top >= kLowTop && top <= kHighTop) || d1 - d0 > A.many) {   // its first draw's outputs say so meanwhile, and keep the maximum
    if (slice == 0 && lane == 0) {
      A.tokens_out[d0] = kLater;
      A.seq_out[d0] = __float_as_int(mx);
    }
    return true;
  }
  if (d0 + turn >= d1) return false;
  const float* row = A.logits + seq * A.vocab;
  Sums<CL>& S = sums[at];
  double end_b, Z;
  block_ends<CL>(S, lane, end_b, Z);
  for (int64_t d = d0 + turn; d < d1; d += kSlices) {
    const double t = static_cast<double>(A.uniforms[d]) * Z;
    int token = A.vocab - 1;                                   // the answer if t is not below the total
    if (t == 0.0) {                                            // the first term that is not 0 at all
      token = first_positive(row, A, S.slice_max, kSlices, static_cast<double>(mx), lane);
    } else if (t < Z) {
      const int b = __ffs(__ballot_sync(0xffffffffu, lane < CL && end_b > t)) - 1;
      const double start = b ? __shfl_sync(0xffffffffu, end_b, max(b - 1, 0)) : 0.0;
      int w = 0;
      double in_front = 0.0;                                   // of slice w in its block
      for (; w < kWarps - 1; ++w) {
        const double e = in_front + S.slice_sum[b * kWarps + w];
        if (start + e > t) break;
        in_front = e;
      }
      const Slice L = slice_of(A, b * kWarps + w);
      const double* seg_end = cg::this_cluster().map_shared_rank(&S, b)->seg_end[w];
      const double before = start + in_front;
      const int n_seg = (L.n_half + 1) >> 1;                   // at most kMaxSegs
      const double end_s = lane < n_seg ? seg_end[lane] : 0.0;
      // (the slice was chosen by start + (in_front + sum), a segment is by (start + in_front) + sum so far: rounded differently,
      //  the slice's end may not be above t here.  Then it is the last segment that added anything - behind it all is masked)
      uint32_t hit = __ballot_sync(0xffffffffu, lane < n_seg && before + end_s > t);
      const double last_end = __shfl_sync(0xffffffffu, end_s, max(n_seg - 1, 0));
      if (!hit) hit = __ballot_sync(0xffffffffu, lane < n_seg && end_s == last_end);
      const int s = __ffs(hit) - 1;
      if (s >= 0) {
        const double in_slice = s ? __shfl_sync(0xffffffffu, end_s, max(s - 1, 0)) : 0.0;
        const int base = L.v0 + s * kSeg;
        Terms T;
        segment_terms<false, VEC>(T, row, A, bank, 0.0, base, min(A.vocab, L.v0 + A.slice), lane);
        token = pick(T, A, base, before + in_slice, t);
      }
    }
    if (lane == 0) {
      A.tokens_out[d] = token;
      A.seq_out[d] = seq;
    }
  }
  return false;
}

template <int CL, bool VEC>
__global__ void __cluster_dims__(CL, 1, 1) __launch_bounds__(kThreads, 1)
branch_sample_kernel(const __grid_constant__ Args A) {
  ss::grid_dependency_enter();
  __shared__ Shared<CL> S;
  cg::cluster_group cl = cg::this_cluster();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int slice = static_cast<int>(cl.block_rank()) * kWarps + warp;
  const Slice L = slice_of(A, slice);
  const double* bank = S.table + (lane & 15);
  // rows with something to draw, in turn (the cluster's blocks agree)
  auto next_row = [&](int64_t r) {
    while (r < A.n_seq && A.draw_offsets[r + 1] <= A.draw_offsets[r]) r += gridDim.x / CL;
    return r;
  };
  const int64_t row0 = A.row0 + static_cast<int64_t>(blockIdx.x / CL);   // (there are no more clusters than rows)
  float first[8];
  load_half<VEC>(A.logits + row0 * A.vocab, L.v0, A.vocab, lane, first);   // in flight while the table is made
  int64_t row = next_row(row0), prev = -1;
  if (row != row0 && row < A.n_seq) load_half<VEC>(A.logits + row * A.vocab, L.v0, A.vocab, lane, first);
  if (tid < kTable) {
    const double e = exp2(static_cast<double>(tid) / kTable);
    S.table[tid * 16] = __hiloint2double(__double2hiint(e) - (tid << 13), __double2loint(e));
  }
  __syncthreads();
  for (int i = tid; i < kTable * 16; i += kThreads)
    if (i & 15) S.table[i] = S.table[i & ~15];
  cl.sync();                                                   // (the table; and every block runs before it is written to)

  int at = 0, prev_at = 0;
  bool later = false;                                          // a row outside the table's range: for when the others are done
  for (;;) {
    double sum = 0.0;
    float mx = -INFINITY;
    const bool more = row < A.n_seq;
    int64_t after = row;
    if (more) {
      const float* p = A.logits + row * A.vocab;
      if (A.fast) {
        sum = slice_sums<VEC>(p, A, bank, S.sums[at].seg_end[warp], L.v0, L.n_half, lane, first, mx);
      } else {
        for (int h = 0; h < L.n_half; ++h) {
          load_half<VEC>(p, L.v0 + h * (kSeg / 2), A.vocab, lane, first);
#pragma unroll
          for (int x = 0; x < 8; ++x) mx = fmaxf(mx, first[x]);
        }
      }
      mx = warp_max(mx);
      after = next_row(row + gridDim.x / CL);
      if (after < A.n_seq) load_half<VEC>(A.logits + after * A.vocab, L.v0, A.vocab, lane, first);
    }
    if (prev >= 0) {
      cluster_wait();
      later |= draws<CL, VEC>(A, S.sums, bank, prev_at, prev, slice, lane);
    }
    if (!more) break;
    publish<CL>(cl, S.sums[at], slice, lane, sum, mx);
    cluster_arrive();
    prev = row;
    prev_at = at;
    at = at == 2 ? 0 : at + 1;
    row = after;
  }
  if (later) {                                                 // (the cluster agrees)
    cl.sync();                                                 // (the marks; and nobody reads the running sums any more)
    for (int64_t r = next_row(row0); r < A.n_seq; r = next_row(r + gridDim.x / CL)) {
      const int64_t d = A.draw_offsets[r];
      if (__ldcg(A.tokens_out + d) != kLater) continue;        // (read in front of row_below's barriers, written behind them)
      row_below<CL, VEC>(A, S.sums[0], S.queue[warp], bank, r, slice, lane, __int_as_float(static_cast<int>(__ldcg(A.seq_out + d))));
    }
  }
  if (CL > 1) cl.sync();                                       // (a block's running sums may still be read by another)
}

// Rows row0 .. n_seq-1, `clusters` at a time.
template <int CL>
static int32_t launch(Args A, bool vec, int row0, int n_seq, int clusters, cudaStream_t st) {
  constexpr int kUnit = kSeg / 2;
  A.slice = (A.vocab + CL * kWarps * kUnit - 1) / (CL * kWarps * kUnit) * kUnit;
  // A draw by itself costs a warp 2.9 us, going through the segments of its slice a second pass over it and 2.5 us a segment.
  // 200 rows of 32000, 128 / 256 / 1024 draws each: 49 / 81 / 269 us one by one, 53 / 58 / 102 by segment (blocks of 1024 threads
  // with the row's sums in shared memory: 68 / 68 / 74); 200 rows of 151936, 256 / 512 / 1024: 109 / 171 / 291 and 175 / 207 / 263
  // (315 / 320 / 331).  Clusters of 4 and 8 blocks have enough warps, one by one is as fast up to 20000 draws, but where most
  // of them would have no slice (4 rows of 300, 4096 draws: 74 and 42).
  const bool idle = static_cast<int64_t>(CL) * kWarps / 2 * A.slice >= A.vocab;
  A.many = CL <= 2 || idle ? CL * kWarps * (4 + A.slice / 384) : INT32_MAX;
  A.row0 = row0;
  A.n_seq = n_seq;
  if (vec)
    SS_LAUNCH((branch_sample_kernel<CL, true>), clusters * CL, kThreads, 0, st, A);
  else
    SS_LAUNCH((branch_sample_kernel<CL, false>), clusters * CL, kThreads, 0, st, A);
  return SS_OK;
}

// Clusters of CL blocks that the current device holds at a time (asked once per device; 74 of 2, 33 of 4, 15 of 8 on 148 SMs).
template <int CL>
static int resident_clusters(bool vec) {
  static std::atomic<int> cached[2][kDeviceSlots];
  const int slot = current_device_slot();
  if (slot >= 0) {
    const int n = cached[vec][slot].load(std::memory_order_relaxed);
    if (n > 0) return n;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(CL);
  cfg.blockDim = dim3(kThreads);
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = CL;
  attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  int n = 0;
  const cudaError_t rc = vec ? cudaOccupancyMaxActiveClusters(&n, branch_sample_kernel<CL, true>, &cfg)
                             : cudaOccupancyMaxActiveClusters(&n, branch_sample_kernel<CL, false>, &cfg);
  if (rc != cudaSuccess || n < 1) {
    (void)cudaGetLastError();
    n = 1;
  }
  if (slot >= 0) cached[vec][slot].store(n, std::memory_order_relaxed);
  return n;
}

}  // namespace sample
}  // namespace ss

extern "C" int32_t ss_branch_sample(const float* logits, const int64_t* draw_offsets, const float* uniforms,
                                    int32_t n_seq, int32_t vocab, float temperature, int32_t* tokens_out,
                                    int64_t* seq_out, void* stream) {
  using namespace ss;
  using namespace ss::sample;
  if (n_seq < 0 || vocab < 1 || !(temperature > 0.f)) return SS_ERR_INVALID_ARG;
  if (vocab > kMaxVocab) return SS_ERR_UNSUPPORTED;
  if (n_seq == 0) return SS_OK;
  if (!logits || !draw_offsets || !uniforms || !tokens_out || !seq_out) return SS_ERR_INVALID_ARG;
  const double T = static_cast<double>(temperature), c = 1.4426950408889634 / T;
  Args A{};
  A.logits = logits;
  A.draw_offsets = draw_offsets;
  A.uniforms = uniforms;
  A.tokens_out = tokens_out;
  A.seq_out = seq_out;
  A.vocab = vocab;
  A.inv_temperature = 1.0 / T;
  A.ck = kTable * c;
  A.ckf = static_cast<float>(A.ck);
  A.lowest = static_cast<float>(kLowest / c);
  A.fast = T >= 1e-3 && T <= 1e6;
  A.lowest_below = kLowest / c;
  const bool vec = reinterpret_cast<uintptr_t>(logits) % 16 == 0 && vocab % 4 == 0;
  cudaStream_t st = as_stream(stream);
  const int sms = sm_count_of_current_device();
  // Whole rounds of one row per SM, then the rows that are left over on clusters as large as fit at once (a cluster that has
  // to wait for another doubles the time: 16 rows 18 us on clusters of 8, of which 15 fit, 13 on clusters of 4).
  // Clusters for all rows cost more than the uneven last round: 250-400 us instead of 186 for 922 rows.
  constexpr int kMaxSlice = kMaxSegs * kSeg * kWarps;           // vocabulary that one block can take (262144)
  const int blocks_min = (vocab + kMaxSlice - 1) / kMaxSlice;   // 1 .. 8
  const int n8 = resident_clusters<8>(vec), n4 = resident_clusters<4>(vec), n2 = resident_clusters<2>(vec);
  auto cluster_size = [&](int rows) { return rows <= n8 ? 8 : rows <= n4 ? 4 : rows <= n2 ? 2 : 1; };
  int whole = blocks_min > 1 ? 0 : n_seq / sms * sms;
  if (blocks_min == 1 && cluster_size(n_seq - whole) == 1) whole = n_seq;
  if (whole > 0) {
    const int32_t rc = launch<1>(A, vec, 0, whole, whole < sms ? whole : sms, st);
    if (rc != SS_OK) return rc;
  }
  const int rest = n_seq - whole;
  if (rest == 0) return SS_OK;
  const int size = cluster_size(rest) > blocks_min ? cluster_size(rest) : blocks_min;
  if (size > 4) return launch<8>(A, vec, whole, n_seq, rest < n8 ? rest : n8, st);
  if (size > 2) return launch<4>(A, vec, whole, n_seq, rest < n4 ? rest : n4, st);
  return launch<2>(A, vec, whole, n_seq, rest < n2 ? rest : n2, st);
}
