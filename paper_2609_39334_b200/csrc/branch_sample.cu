// ss_branch_sample: the sampling half of on-demand branching (paper, Section "Computation Deduplication"): a
// sequence with potential size n draws n next tokens as independent trials from ONE logits row; equal draws are
// grouped afterwards with ss_dedup_paths on (sequence, token) pairs.
//
// The token decision is that of fp64 (it agrees with a plain fp64 CPU evaluation except for draws within
// ~1e-15 of a boundary), one exponential per logit.  A row is split over the 16 warps of a block, or of a CLUSTER of
// 2, 4 or 8 blocks when there are too few rows to give every SM one: each warp has one contiguous slice, and the slice sums
// meet in (distributed) shared memory.  Nothing is read twice but the 512 tokens around each draw, and the row of a draw that fp32
// sums leave open (below).
//   1. every warp sums 2^(logit_v * c), c = log2(e) / temperature, over its slice in segments of 512 tokens and keeps
//      the running sum at every segment's end (shared memory)
//   2. the slice sums are written to every block of the cluster
//   3. each draw is a warp's: it finds the slice that holds u * Z from the slice sums, the
//      segment from the running sums of the slice's owner, evaluates the segment again with a warp scan, and writes the
//      token
// A cluster that handles several rows takes step 1 of the next row before step 3 of the current one, between the two halves
// of a split barrier; a block that handles rows by itself has four warps for step 3 alone.
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
//
// Those hold the issue slots: 32 logits take ~30 clocks of a sub-partition, 922 rows of 151936 120 us where the 560 MB take 85.  So
// where there are many rows with few draws, blocks add them up in fp32 (quick_sums: 7 packed instructions a logit, eight terms at a
// time before fp64).  A quick sum is within 3.2e-7 of the exact one, proven; a draw whose target is not further than
// that from the two ends of its token (1.5 % of them) is marked and made again by the table, its whole row, in the launch
// that takes the rows that are left over.  No token is other than the table's.
// Bound now: HBM latency and issue slots about equally (86 us with the arithmetic taken out).  Measured, the call: 922 rows, 1362
// draws 184 us by the table -> 130 (rows 97, marked draws and left-over rows 33), of it 20 by adding up four segments' sums over
// the warp at once; 16 rows 12.4.
#include <cooperative_groups.h>
#include <stdlib.h>

#include "common.cuh"
#include "umma.cuh"

namespace ss {
namespace sample {

namespace cg = cooperative_groups;

constexpr int kThreads = 512;                                 // one block per SM (128 registers a thread)
constexpr int kWarps = kThreads / 32;
constexpr int kSeg = 512;                                     // tokens per segment: 16 per lane, 4 x 128 bits
constexpr int kMaxSegs = 32;                                  // per slice
constexpr int kMaxVocab = 2097152;
constexpr int kTable = 128;
constexpr int kLater = -1, kUnsure = -2, kTaken = -3;         // not tokens
// Blocks that take rows by themselves (branch_rows_kernel)
constexpr int kDrawWarps = 4;                                 // behind the kWarps that add up
constexpr int kRowThreads = kThreads + 32 * kDrawWarps;       // (96 registers a thread)
constexpr int kStages = 4;                                    // segments of a warp in shared memory or on their way there
constexpr int kRingBytes = kWarps * kStages * kSeg * 4;
constexpr int kSums = 3;                                      // rows whose sums are held at a time
constexpr double kQuickError = 3.2e-7;                        // of the quick sums, see quick_sums
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
  float c_hi, c_lo, inv_c;     // log2(e) / temperature in two parts, and its reciprocal
  int quick_draws;             // draws of a row up to which its sums are quick ones
  int whole_draws;             // rows with more draws are left to the clusters as a whole
  int first_idle;              // clusters from here on have no row of their own and take marked draws
  double lowest_below;         // the same for l - dm
  bool fast;                   // the temperature allows sums that are not relative to the row's maximum
#ifdef SS_CHECKED
  bool give_up;                // waits between warps are to be taken for run out
#endif
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
  int pick, taken;                     // see next_unsure
};
struct RowShared {                     // of branch_rows_kernel
  uint64_t full[kSums], free[kSums];   // a row's sums are there; its draws are made
  int abort_flag, later;
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
// ---- rows that a block takes by itself -------------------------------------------------------------------------------
// Every lane copies what it reads itself (16 logits a segment), so that nothing has to be synchronised: 3 segments of each
// warp, 96 KB an SM, are in flight whatever the arithmetic does.
template <bool VEC>
__device__ __forceinline__ void request(uint32_t dst, const float* __restrict__ row, int base, int end, int lane) {
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int v = base + 128 * j + 4 * lane;
    const uint32_t d = dst + 512 * j;
    if (VEC) {
      if (v < end)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(row + v) : "memory");
      else
        asm volatile("st.shared.v4.b32 [%0], {%1, %1, %1, %1};" ::"r"(d), "r"(0xff800000u) : "memory");   // -inf
    } else {
#pragma unroll
      for (int x = 0; x < 4; ++x) {
        if (v + x < end)
          asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(d + 4 * x), "l"(row + v + x) : "memory");
        else
          asm volatile("st.shared.b32 [%0], %1;" ::"r"(d + 4 * x), "r"(0xff800000u) : "memory");
      }
    }
  }
}
// A whole segment, `src`: the lane's first logit of it.
__device__ __forceinline__ void request_whole(uint32_t dst, const float* __restrict__ src) {
#pragma unroll
  for (int j = 0; j < 4; ++j)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + 512 * j), "l"(src + 128 * j) : "memory");
}
__device__ __forceinline__ void read_segment(uint32_t src, float (&l)[16]) {
#pragma unroll
  for (int j = 0; j < 4; ++j)
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(l[4 * j]), "=f"(l[4 * j + 1]), "=f"(l[4 * j + 2]), "=f"(l[4 * j + 3])
                 : "r"(src + 512 * j) : "memory");
}
__device__ __forceinline__ float max_nan(float a, float b) {
  float d;
  asm("max.NaN.f32 %0, %1, %2;" : "=f"(d) : "f"(a), "f"(b));
  return d;
}
// A lane's sum of a segment by the table, and its largest logit so far.
__device__ __forceinline__ double exact_sums(float (&l)[16], const Args& A, const double* bank, float& mx) {
  double s0 = 0.0, s1 = 0.0;
#pragma unroll
  for (int h = 0; h < 16; h += 8) {
    float mn = l[h];
#pragma unroll
    for (int x = h; x < h + 8; ++x) { mx = fmaxf(mx, l[x]); mn = fminf(mn, l[x]); }
    if (__any_sync(0xffffffffu, !(mn >= A.lowest))) {          // masked tokens, or past the end (a NaN stays one)
#pragma unroll
      for (int x = h; x < h + 8; ++x) l[x] = max_nan(l[x], A.lowest);
    }
#pragma unroll
    for (int x = h; x < h + 8; x += 2) {
      s0 += exp2_table(l[x], A, bank);
      s1 += exp2_table(l[x + 1], A, bank);
    }
  }
  return s0 + s1;
}

// Sums of four values over the warp at once (18 instructions instead of 60): lane l gets that of v[l / 8].
__device__ __forceinline__ double warp_sums_4(const double (&v)[4], int lane) {
  const bool up = (lane & 16) != 0, right = (lane & 8) != 0;
  const double a = (up ? v[2] : v[0]) + __shfl_xor_sync(0xffffffffu, up ? v[0] : v[2], 16);
  const double b = (up ? v[3] : v[1]) + __shfl_xor_sync(0xffffffffu, up ? v[1] : v[3], 16);
  double c = (right ? b : a) + __shfl_xor_sync(0xffffffffu, right ? a : b, 8);
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
  return c;
}

// A lane's sum of a segment in fp32, two logits at a time, relative to a power of two 2^e0 that the lane moves when a logit exceeds
// it by 2^60.
// l * c = n + f with |f| <= 1/2: n from a sum whose low bits are the integer, f exactly by an FMA with the high part of c (one
// rounding to 2^-26) and one with the low part; 2^f by a polynomial of degree 6 (minimax of the relative error on |f| <=
// 0.5002, coefficients rounded: 1.6e-8); n into the exponent by an integer addition.  A term is within 1.21e-7: 1.6e-8, 2.1e-8
// from f, 2.4e-8 from the polynomial's inner roundings and 6e-8 from its last one.  Eight terms are added pairwise (three
// roundings, 1.79e-7) and go to fp64 from there: a sum of any of them is within kQuickError of the exact one.  Terms below
// 2^(e0 - 124) count as that, 2^-124 of the lane's largest and less.
struct QuickState {
  float mx, e0, low, shift;
};
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pack2(float a, float b) { f32x2 r; asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b)); return r; }
__device__ __forceinline__ void unpack2(f32x2 v, float& a, float& b) { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v)); }
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) { f32x2 r; asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c)); return r; }
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) { f32x2 r; asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b)); return r; }
__device__ __forceinline__ f32x2 both(float a) { return pack2(a, a); }
__device__ __forceinline__ void quick_base(QuickState& q, const Args& A, float e0) {
  q.e0 = e0;
  q.low = (e0 - 124.f) * A.inv_c;
  q.shift = 12582912.f - e0;                                   // 1.5 * 2^23
}
__device__ __forceinline__ f32x2 quick_terms(float l0, float l1, const QuickState& q, const Args& A) {
  const f32x2 l = pack2(fmaxf(l0, q.low), fmaxf(l1, q.low)), c_hi = both(A.c_hi);
  const f32x2 nb = fma2(l, c_hi, both(q.shift));               // bits: 0x4b400000 + (n - e0)
  f32x2 f = fma2(l, c_hi, fma2(nb, both(-1.f), both(q.shift)));
  f = fma2(l, both(A.c_lo), f);
  f32x2 p = fma2(f, both(0.00015353319759014994f), both(0.0013398926239460707f));
  p = fma2(p, f, both(0.009618437848985195f));
  p = fma2(p, f, both(0.055503323674201965f));
  p = fma2(p, f, both(0.24022647738456726f));
  p = fma2(p, f, both(0.6931471824645996f));
  p = fma2(p, f, both(1.f));
  float p0, p1, n0, n1;
  unpack2(p, p0, p1);
  unpack2(nb, n0, n1);
  return pack2(__int_as_float(__float_as_int(p0) + (__float_as_int(n0) << 23)), __int_as_float(__float_as_int(p1) + (__float_as_int(n1) << 23)));
}
__device__ __forceinline__ double quick_sums(const float (&l)[16], const Args& A, QuickState& q) {
  float top = l[0];
#pragma unroll
  for (int x = 1; x < 16; ++x) top = max_nan(top, l[x]);
  q.mx = max_nan(q.mx, top);
  const float te = top * A.c_hi;
  if (te > q.e0 + 60.f) quick_base(q, A, rintf(fminf(te, 2000.f)));   // (such a row is out of range anyway)
  const int e0 = __float2int_rn(q.e0) << 20;
  double s = 0.0;
#pragma unroll
  for (int h = 0; h < 16; h += 8) {
    const f32x2 t = add2(add2(quick_terms(l[h], l[h + 1], q, A), quick_terms(l[h + 2], l[h + 3], q, A)),
                         add2(quick_terms(l[h + 4], l[h + 5], q, A), quick_terms(l[h + 6], l[h + 7], q, A)));
    float a, b;
    unpack2(t, a, b);
    const double d = static_cast<double>(a + b);
    s += __hiloint2double(__double2hiint(d) + e0, __double2loint(d));
  }
  return s;
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
// The token of target t, which lies in the segment at `base`; `before`: the sum in front of it.  With BOUNDS also the sums up to
// the token and with it (from > to where t is above the segment's terms).
template <bool BOUNDS = false>
__device__ __forceinline__ int pick(const Terms& T, const Args& A, int base, double before, double t, double* from = nullptr,
                                    double* to = nullptr) {
  if (BOUNDS) { *from = INFINITY; *to = 0.0; }
  int token = -1;                                              // if rounding leaves t above everything: the last that counts
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const uint32_t some = __ballot_sync(0xffffffffu, T.run[j] > kTiny);
    const uint32_t over = __ballot_sync(0xffffffffu, T.run[j] > kTiny && before + T.incl[j] > t);
    if (some) {
      const int f = over ? __ffs(over) - 1 : 31 - __clz(some);
      double c = before + (T.incl[j] - T.run[j]);
      int hit = -1, tail = 0;
      double below = INFINITY, above = 0.0;
#pragma unroll
      for (int x = 0; x < 4; ++x) {
        const double start = c;
        c += T.e[j][x];
        if (T.e[j][x] > kTiny) {
          tail = x;
          if (hit < 0 && c > t) {
            hit = x;
            below = start;
            above = c;
          }
        }
      }
      token = base + 128 * j + 4 * f + __shfl_sync(0xffffffffu, hit < 0 ? tail : hit, f);
      if (over) {
        if (BOUNDS) {
          *from = __shfl_sync(0xffffffffu, below, f);
          *to = __shfl_sync(0xffffffffu, above, f);
        }
        return token;
      }
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

// A row that is left to the clusters: its first draw is marked, the others are none of theirs.
__device__ __forceinline__ void mark_whole(const Args& A, int64_t seq, int64_t d0, int64_t d1, int lane) {
  for (int64_t d = d0 + lane; d < d1; d += 32) {
    A.tokens_out[d] = d == d0 ? kUnsure : kTaken;
    A.seq_out[d] = seq;
  }
}

// Draws d0 + turn, d0 + turn + turns, ... below d1 of row `seq`; `at`: which of `sums` holds the row.  True, with nothing drawn,
// if the row is outside the table's range or has many draws (all that draw from it agree).
// QUICK: the sums may be quick ones (`quick`), each within kQuickError of the exact one.  The terms of the segment that holds the
// target are exact ones, so a token whose sums lie further from the target than the errors of both can add up to is the exact
// sums' token too; a draw for which that cannot be said is marked, and taken by a launch that adds up its row by the table.
template <int CL, bool VEC, bool QUICK>
__device__ __forceinline__ bool draws(const Args& A, Sums<CL>* sums, const double* bank, int at, int64_t seq, int64_t d0, int64_t d1,
                                      int turn, int turns, bool quick, int lane) {
  constexpr int kSlices = CL * kWarps;
  if (QUICK && d1 - d0 > A.many) {
    if (turn == 0) mark_whole(A, seq, d0, d1, lane);
    return false;
  }
  float mx = -INFINITY;
  for (int i = lane; i < kSlices; i += 32) mx = fmaxf(mx, sums[at].slice_max[i]);
  mx = warp_max(mx);
  const float top = mx * A.ckf * (1.f / kTable);
  if (!(A.fast && top >= kLowTop && top <= kHighTop) || (!QUICK && d1 - d0 > A.many)) {   // its first draw's outputs say so meanwhile, and keep the maximum
    if (turn == 0 && lane == 0) {
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
  for (int64_t d = d0 + turn; d < d1; d += turns) {
    const double t = static_cast<double>(A.uniforms[d]) * Z;
    int token = A.vocab - 1;                                   // the answer if t is not below the total
    bool sure = !(QUICK && quick) || Z != Z;
    if (t == 0.0) {                                            // the first term that is not 0 at all
      token = first_positive(row, A, S.slice_max, kSlices, static_cast<double>(mx), lane);
      sure = true;
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
        if (QUICK) {
          double from, to;
          token = pick<true>(T, A, base, before + in_slice, t, &from, &to);
          const double slack = t * (2.05 * kQuickError);
          sure = sure || (from <= t - slack && to > t + slack);
        } else {
          token = pick(T, A, base, before + in_slice, t);
        }
      }
    }
    if (lane == 0) {
      A.tokens_out[d] = sure ? token : kUnsure;
      A.seq_out[d] = seq;
    }
  }
  return false;
}

template <int THREADS>
__device__ __forceinline__ void make_table(double* table) {
  const int tid = threadIdx.x;
  if (tid < kTable) {
    const double e = exp2(static_cast<double>(tid) / kTable);
    table[tid * 16] = __hiloint2double(__double2hiint(e) - (tid << 13), __double2loint(e));
  }
  __syncthreads();
#pragma unroll
  for (int i0 = 0; i0 < kTable * 16; i0 += THREADS) {
    const int i = i0 + tid;
    if ((THREADS == kThreads || i < kTable * 16) && (i & 15)) table[i] = table[i & ~15];
  }
}

// What is worked on in turn: draws d0 .. d1 - 1 of `row` (-1: nothing).
struct Work {
  int64_t row, d0, d1;
};
// The next row with something to draw.
__device__ __forceinline__ Work next_row(const Args& A, int64_t r, int step) {
  for (; r < A.n_seq; r += step) {
    const int64_t d0 = A.draw_offsets[r], d1 = A.draw_offsets[r + 1];
    if (d1 > d0) return Work{r, d0, d1};
  }
  return Work{-1, 0, 0};
}

// A row per block at a time.  kWarps warps add up the rows one after the other, quick where a row has few draws; kDrawWarps warps
// make the draws of the rows whose sums are complete (a draw takes 2.9 us, and a warp that made it between two rows held up all
// others at the end of the next).  Four warps make as many draws in the time of a row as it has thousands of tokens, about: a row
// with more than a few times that is left to the clusters, which have 32 warps or more (592 rows of 151936, one draw each but 256
// of one row: 209 us if its block makes them, 102 so).  The waits are between warps of a block and bounded; the call has no status to
// say that one ran out, so the block then takes all of its rows again, by row_below with its hardware barriers.
template <bool VEC>
__global__ void __launch_bounds__(kRowThreads, 1) branch_rows_kernel(const __grid_constant__ Args A) {
  ss::grid_dependency_enter();
  extern __shared__ __align__(16) float ring[];
  __shared__ Shared<1> S;
  __shared__ RowShared C;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, step = gridDim.x;
  const double* bank = S.table + (lane & 15);
  volatile int* abort_flag = &C.abort_flag;
  const int64_t row0 = A.row0 + static_cast<int64_t>(blockIdx.x);
  if (tid == 0) {
    for (int i = 0; i < kSums; ++i) {
      umma::mbar_init(&C.full[i], kWarps);
      umma::mbar_init(&C.free[i], kDrawWarps);
    }
    C.abort_flag = C.later = 0;
    umma::fence_barrier_init();
  }
  const Slice L = slice_of(A, min(warp, kWarps - 1));
  const int n_seg = (L.n_half + 1) >> 1, end = min(A.vocab, L.v0 + A.slice);
  const int n_whole = end > L.v0 ? (end - L.v0) / kSeg : 0;    // segments without an end
  const uint32_t my_ring = umma::smem_u32(ring) + (min(warp, kWarps - 1) * kStages * kSeg + 4 * lane) * 4;
  Work now = next_row(A, row0, step), req = now;
  int req_seg = 0, req_stage = 0, stage = 0;
  // The requests run kStages - 1 segments ahead of the sums, into the rows that follow; a group is closed for every segment, asked
  // for or not.
  auto request_next = [&]() {
    if (req.row >= 0 && n_seg > 0) {
      const uint32_t dst = my_ring + req_stage * (kSeg * 4);
      if (VEC && req_seg < n_whole)
        request_whole(dst, A.logits + (req.row * A.vocab + L.v0 + req_seg * kSeg + 4 * lane));
      else
        request<VEC>(dst, A.logits + req.row * A.vocab, L.v0 + req_seg * kSeg, end, lane);
      if (++req_seg == n_seg) {
        req_seg = 0;
        req = next_row(A, req.row + step, step);
      }
    }
    req_stage = req_stage == kStages - 1 ? 0 : req_stage + 1;
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  if (warp < kWarps) {
#pragma unroll 1
    for (int x = 0; x < kStages - 1; ++x) request_next();
  }
  make_table<kRowThreads>(S.table);
  __syncthreads();

  uint32_t count = 0;                                          // rows so far: their sums lie in turn in the kSums places
  auto wait = [&](uint64_t* bar, uint32_t turn) {
#ifdef SS_CHECKED
    if (A.give_up && warp >= kWarps && count == 1) *abort_flag = 1;
    if (A.give_up && __any_sync(0xffffffffu, *abort_flag)) return false;
#endif
    return __all_sync(0xffffffffu, umma::mbar_wait(bar, turn & 1, abort_flag)) != 0;   // (a warp leaves as a whole)
  };
  if (warp < kWarps) {
    for (; now.row >= 0; ++count) {
      const int at = count % kSums;
      if (count >= kSums && !wait(&C.free[at], count / kSums - 1)) break;
      const bool quick = A.fast && now.d1 - now.d0 <= A.quick_draws;
      double sum = 0.0;
      float mx = -INFINITY;
      QuickState q;
      q.mx = -INFINITY;
      quick_base(q, A, -330.f);
      auto next_segment = [&](float (&l)[16]) {
        request_next();
        asm volatile("cp.async.wait_group %0;" ::"n"(kStages - 1) : "memory");
        read_segment(my_ring + stage * (kSeg * 4), l);
        stage = stage == kStages - 1 ? 0 : stage + 1;
      };
      if (quick) {
        double mine = 0.0;                                     // of segment `lane`
#pragma unroll 1
        for (int s = 0; s < n_seg; s += 4) {
          double v[4];
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            v[k] = 0.0;
            if (s + k < n_seg) {
              float l[16];
              next_segment(l);
              v[k] = quick_sums(l, A, q);
            }
          }
          const double four = __shfl_sync(0xffffffffu, warp_sums_4(v, lane), (lane & 3) * 8);
          if ((lane & ~3) == s) mine = four;
        }
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const double y = __shfl_up_sync(0xffffffffu, mine, o);
          if (lane >= o) mine += y;
        }
        if (lane < n_seg) S.sums[at].seg_end[warp][lane] = mine;
        sum = __shfl_sync(0xffffffffu, mine, 31);
      } else {
#pragma unroll 1
        for (int s = 0; s < n_seg; ++s) {
          float l[16];
          next_segment(l);
          if (A.fast) {
            sum += warp_sum_d(exact_sums(l, A, bank, mx));
            if (lane == 0) S.sums[at].seg_end[warp][s] = sum;
          } else {
#pragma unroll
            for (int x = 0; x < 16; ++x) mx = fmaxf(mx, l[x]);
          }
        }
      }
      if (quick) {
        if (__any_sync(0xffffffffu, q.mx != q.mx)) sum = __longlong_as_double(0x7ff8000000000000ll);   // (as the exact sums would be)
        mx = q.mx;
      }
      mx = warp_max(mx);
      if (lane == 0) {
        S.sums[at].slice_sum[warp] = sum;
        S.sums[at].slice_max[warp] = mx;
      }
      __syncwarp();                                            // (every lane has written a segment's end)
      if (lane == 0) umma::mbar_arrive(&C.full[at]);
      now = next_row(A, now.row + step, step);
    }
  } else {
    bool later = false;                                        // a row outside the table's range: for when the others are done
    for (; now.row >= 0; ++count) {
      const int at = count % kSums;
      if (!wait(&C.full[at], count / kSums)) break;
      __syncwarp();
      const int turn = (warp + static_cast<int>(now.row)) % kDrawWarps;
      later |= draws<1, VEC, true>(A, S.sums, bank, at, now.row, now.d0, now.d1, turn, kDrawWarps,
                                   A.fast && now.d1 - now.d0 <= A.quick_draws, lane);
      __syncwarp();
      if (lane == 0) umma::mbar_arrive(&C.free[at]);
      now = next_row(A, now.row + step, step);
    }
    if (later && lane == 0) C.later = 1;
  }
  __syncthreads();                                             // (the marks; and nobody reads the running sums any more)
  if (C.abort_flag) {                                          // a wait ran out
    asm volatile("cp.async.wait_all;" ::: "memory");
    for (int64_t r = row0 + static_cast<int64_t>(step) * warp; r < A.n_seq; r += static_cast<int64_t>(step) * (kRowThreads / 32)) {
      const int64_t d = A.draw_offsets[r];
      if (A.draw_offsets[r + 1] <= d) continue;
      float mx = -INFINITY;
      for (int v = lane; v < A.vocab; v += 32) mx = fmaxf(mx, __ldg(A.logits + r * A.vocab + v));
      mx = warp_max(mx);
      if (lane == 0) {
        A.tokens_out[d] = kLater;
        A.seq_out[d] = __float_as_int(mx);
      }
    }
    if (tid == 0) C.later = 1;
    __syncthreads();
  }
  if (C.later) {
    for (Work r = next_row(A, row0, step); r.row >= 0; r = next_row(A, r.row + step, step)) {
      if (__ldcg(A.tokens_out + r.d0) != kLater) continue;     // (read in front of row_below's barriers, written behind them)
      if (warp < kWarps) {
        row_below<1, VEC>(A, S.sums[0], S.queue[warp], bank, r.row, warp, lane, __int_as_float(static_cast<int>(__ldcg(A.seq_out + r.d0))));
      } else {                                                 // (its two barriers)
        cg::this_cluster().sync();
        cg::this_cluster().sync();
      }
    }
  }
}

// The cluster's next marked draw among those of the rows in front of this launch's: its first block looks at 4096 draws at a time
// and takes the first mark behind a place of the cluster's own, until one is its.
template <int CL>
__device__ __forceinline__ Work next_unsure(cg::cluster_group& cl, const Args& A, Shared<CL>& S, int64_t& scanned, int cluster, int n_clusters) {
  constexpr int kScan = 8 * kThreads;
  const int tid = threadIdx.x;
  const int64_t first = A.draw_offsets[0], count = A.draw_offsets[A.row0] - first;
  if (cl.block_rank() == 0) {
    int64_t found = -1;
    while (found < 0 && scanned < count) {
      const int left = static_cast<int>(count - scanned < kScan ? count - scanned : kScan);
      const int start = static_cast<int>(static_cast<int64_t>(cluster - A.first_idle) * left / (n_clusters - A.first_idle));
      if (tid == 0) S.pick = INT32_MAX;
      __syncthreads();
      int key = INT32_MAX;
#pragma unroll
      for (int k = 0; k < kScan / kThreads; ++k) {
        const int i = k * kThreads + tid;
        if (i < left && __ldcg(A.tokens_out + first + scanned + i) == kUnsure) key = min(key, (i - start) & (kScan - 1));
      }
      if (key != INT32_MAX) atomicMin(&S.pick, key);
      __syncthreads();
      const int pick = S.pick;
      if (pick == INT32_MAX) {
        scanned += kScan;
      } else {
        const int64_t d = first + scanned + ((pick + start) & (kScan - 1));
        if (tid == 0) S.taken = atomicCAS(A.tokens_out + d, kUnsure, kTaken) == kUnsure ? 1 : 0;
        __syncthreads();
        if (S.taken) found = d - first;
      }
      __syncthreads();
    }
    if (tid < CL) cl.map_shared_rank(&S, tid)->taken = static_cast<int>(found);
  }
  cl.sync();
  const int i = S.taken;
  cl.sync();                                                   // (it is written to again)
  if (i < 0) return Work{-1, 0, 0};
  const int64_t row = __ldcg(A.seq_out + first + i), d0 = A.draw_offsets[row], d1 = A.draw_offsets[row + 1];
  return d1 - d0 > A.whole_draws ? Work{row, d0, d1} : Work{row, first + i, first + i + 1};
}

// A row per cluster at a time; UNSURE: then the draws and rows that the launch before this one has marked.
template <int CL, bool VEC, bool UNSURE>
__global__ void __cluster_dims__(CL, 1, 1) __launch_bounds__(kThreads, 1)
branch_sample_kernel(const __grid_constant__ Args A) {
  ss::grid_dependency_enter();
  __shared__ Shared<CL> S;
  cg::cluster_group cl = cg::this_cluster();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int slice = static_cast<int>(cl.block_rank()) * kWarps + warp;
  const Slice L = slice_of(A, slice);
  const double* bank = S.table + (lane & 15);
  const int cluster = blockIdx.x / CL, n_clusters = gridDim.x / CL;
  const int64_t row0 = A.row0 + static_cast<int64_t>(cluster);
  float first[8];
  if (row0 < A.n_seq) load_half<VEC>(A.logits + row0 * A.vocab, L.v0, A.vocab, lane, first);   // in flight while the table is made
  // rows with something to draw, in turn (the cluster's blocks agree)
  auto next_row = [&](int64_t r) {
    while (r < A.n_seq && A.draw_offsets[r + 1] <= A.draw_offsets[r]) r += n_clusters;
    return r;
  };
  int64_t row = next_row(row0), prev = -1;
  if (row != row0 && row < A.n_seq) load_half<VEC>(A.logits + row * A.vocab, L.v0, A.vocab, lane, first);
  make_table<kThreads>(S.table);
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
      after = next_row(row + n_clusters);
      if (after < A.n_seq) load_half<VEC>(A.logits + after * A.vocab, L.v0, A.vocab, lane, first);
    }
    if (prev >= 0) {
      cluster_wait();
      later |= draws<CL, VEC, false>(A, S.sums, bank, prev_at, prev, A.draw_offsets[prev], A.draw_offsets[prev + 1],
                                     static_cast<int>((slice + prev) % (CL * kWarps)), CL * kWarps, false, lane);
    }
    if (!more) break;
    publish<CL>(cl, S.sums[at], slice, lane, sum, mx);
    cluster_arrive();
    prev = row;
    prev_at = at;
    at = at == 2 ? 0 : at + 1;
    row = after;
  }
  if (later) cl.sync();                                        // (the marks; and nobody reads the running sums any more.  The cluster agrees)
  int64_t r = later ? next_row(row0) : A.n_seq, scanned = 0;
  for (;;) {                                                   // rows that wait for their maximum, then what the launch before has marked
    int64_t below = -1, d0 = 0;
    if (r < A.n_seq) {
      d0 = A.draw_offsets[r];
      if (__ldcg(A.tokens_out + d0) == kLater) below = r;      // (read in front of row_below's barriers, written behind them)
      r = next_row(r + n_clusters);
    } else if (UNSURE && cluster >= A.first_idle) {
      const Work now = next_unsure<CL>(cl, A, S, scanned, cluster, n_clusters);
      if (now.row < 0) break;
      const float* p = A.logits + now.row * A.vocab;
      float mx;
      load_half<VEC>(p, L.v0, A.vocab, lane, first);
      const double sum = slice_sums<VEC>(p, A, bank, S.sums[0].seg_end[warp], L.v0, L.n_half, lane, first, mx);
      publish<CL>(cl, S.sums[0], slice, lane, sum, warp_max(mx));
      cl.sync();
      if (draws<CL, VEC, false>(A, S.sums, bank, 0, now.row, now.d0, now.d1, slice, CL * kWarps, false, lane)) below = now.row;
      d0 = now.d0;
      cl.sync();
    } else {
      break;
    }
    if (below >= 0)
      row_below<CL, VEC>(A, S.sums[0], S.queue[warp], bank, below, slice, lane, __int_as_float(static_cast<int>(__ldcg(A.seq_out + d0))));
  }
  if (CL > 1) cl.sync();                                       // (a block's running sums may still be read by another)
}

template <bool VEC>
static bool ring_ready() {
  static bool configured[kDeviceSlots] = {false};
  const int slot = current_device_slot();
  if (slot >= 0 && configured[slot]) return true;
  if (cudaFuncSetAttribute(branch_rows_kernel<VEC>, cudaFuncAttributeMaxDynamicSharedMemorySize, kRingBytes) != cudaSuccess) {
    (void)cudaGetLastError();
    return false;
  }
  if (slot >= 0) configured[slot] = true;
  return true;
}

// Rows 0 .. n_seq-1, one per block at a time; a launch of clusters has to follow.
// Quick sums leave 1.5 % of the draws of a row of 151936 ordinary logits open (9 % if the logits are all equal), each of which
// costs another pass over its row, by the table: worth it up to 16 draws of such a row.
static int32_t launch_rows(Args A, bool vec, int n_seq, int blocks, cudaStream_t st) {
  constexpr int kUnit = kSeg / 2;
  A.slice = (A.vocab + kWarps * kUnit - 1) / (kWarps * kUnit) * kUnit;
  A.many = A.whole_draws;
  A.quick_draws = 2500000 / A.vocab;
  A.n_seq = n_seq;
  if (!(vec ? ring_ready<true>() : ring_ready<false>())) return SS_ERR_CUDA;
  if (vec)
    SS_LAUNCH(branch_rows_kernel<true>, blocks, kRowThreads, kRingBytes, st, A);
  else
    SS_LAUNCH(branch_rows_kernel<false>, blocks, kRowThreads, kRingBytes, st, A);
  return SS_OK;
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
  const bool unsure = CL > 1 && A.first_idle != INT32_MAX;
  if (vec && unsure)
    SS_LAUNCH((branch_sample_kernel<CL, true, (CL > 1)>), clusters * CL, kThreads, 0, st, A);
  else if (vec)
    SS_LAUNCH((branch_sample_kernel<CL, true, false>), clusters * CL, kThreads, 0, st, A);
  else if (unsure)
    SS_LAUNCH((branch_sample_kernel<CL, false, (CL > 1)>), clusters * CL, kThreads, 0, st, A);
  else
    SS_LAUNCH((branch_sample_kernel<CL, false, false>), clusters * CL, kThreads, 0, st, A);
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
  const cudaError_t rc = vec ? cudaOccupancyMaxActiveClusters(&n, branch_sample_kernel<CL, true, true>, &cfg)
                             : cudaOccupancyMaxActiveClusters(&n, branch_sample_kernel<CL, false, true>, &cfg);
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
  return ss_branch_sample_upto(logits, draw_offsets, uniforms, n_seq, vocab, temperature, tokens_out, seq_out, -1, stream);
}

extern "C" int32_t ss_branch_sample_upto(const float* logits, const int64_t* draw_offsets, const float* uniforms,
                                         int32_t n_seq, int32_t vocab, float temperature, int32_t* tokens_out,
                                         int64_t* seq_out, int64_t max_draws, void* stream) {
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
  A.c_hi = static_cast<float>(c);
  A.c_lo = static_cast<float>(c - static_cast<double>(A.c_hi));
  A.inv_c = static_cast<float>(1.0 / c);
#ifdef SS_CHECKED
  A.give_up = getenv("SS_GIVE_UP") != nullptr;
#endif
  A.first_idle = INT32_MAX;
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
  // fp32 sums save a block 0.06 us per 1000 tokens and cost a launch for the draws that they leave open, and four warps make a row's
  // draws instead of sixteen: for calls with many tokens a block and, by the caller's bound, few draws a row.  Table -> fp32, us,
  // rows x vocabulary, draws of a row: 922 x 151936, 1: 184 -> 121, 4: 185 -> 151; 740 x 128256, 4: 118 -> 105; 740 x 100352, 1: 95 ->
  // 78; 592 x 100352, 1: 77 -> 68; 888 x 65536, 1: 80 -> 64; 2400 x 32000, 2: 131 -> 97.  On the other side 740 x 65536, 1: 66 -> 67;
  // 592 x 65536, 1: 55 -> 61; 444 x 100352, 1: 60 -> 65; 740 x 100352, 4: 95 -> 106; 922 x 151936, 16: 196 -> 287; 148 x 151936, 1:
  // 30 -> 40, 148 x 16384, 1: 8 -> 20.  Smaller vocabularies gain little at any number of rows (2400 x 16384, 1: 89 -> 85).
  const int64_t tokens = static_cast<int64_t>(whole / sms) * vocab;   // of a block
  // A few rows left over go to clusters of 8 otherwise, too few of them for the marked draws (1490 x 151936, 3: 286 -> 402 us with them,
  // 260 with clusters of 4): with less than five rounds in front of them the table keeps them.
  const bool few_left = n_seq > whole && n_seq - whole <= n8;
  const bool rows = max_draws >= 0 && A.fast && vocab >= 32000 && tokens >= 390000 && (!few_left || whole / sms >= 5) &&
                    max_draws <= static_cast<int64_t>(n_seq) * (tokens >= 1000000 ? 5 : tokens >= 605000 ? 4 : tokens >= 500000 ? 3 : 2);
  if (rows) A.whole_draws = vocab >> 12 > 16 ? vocab >> 12 : 16;
  if (whole > 0) {
    const int blocks = whole < sms ? whole : sms;
    const int32_t rc = rows ? launch_rows(A, vec, whole, blocks, st) : launch<1>(A, vec, 0, whole, blocks, st);
    if (rc != SS_OK) return rc;
  }
  const int rest = n_seq - whole;
  if (rest == 0 && !rows) return SS_OK;
  int size = rest ? cluster_size(rest) : 4;
  if (rows && size > 4) size = 4;
  if (size < blocks_min) size = blocks_min;
  const int resident = size > 4 ? n8 : size > 2 ? n4 : n2;
  int clusters = rest < resident ? rest : resident;
  if (rows) {                                                   // marked draws: by the clusters without a row, unless they are few
    clusters = resident;
    A.first_idle = (resident - rest) * 4 >= resident ? rest : 0;
  }
  if (size > 4) return launch<8>(A, vec, whole, n_seq, clusters, st);
  if (size > 2) return launch<4>(A, vec, whole, n_seq, clusters, st);
  return launch<2>(A, vec, whole, n_seq, clusters, st);
}
