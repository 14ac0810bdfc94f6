// score_kernel.cu - fused per-position scoring over the vocabulary and top-k
// seed selection.
//
// Per row (one CTA, or one cluster, per row; the row streamed once from HBM):
//   greedy token y_hat = argmax p and confidence c = max p       (Section 3)
//   entropy H = -sum p ln p                                       (Section 6.1)
//   uncertainty u = -log p(y), Score = u (1 + d_in)/(1 + d_out)   (Section 5.3)
// with p = softmax(logits) at temperature 1. Each thread keeps, for its share
// of the row, the running maximum m (exact bf16 compare, first index kept),
// Z = sum 2^t and S = sum t 2^t with t = x log2(e) - m log2(e), Kahan
// compensated; partials are re-referenced to the row maximum and summed across
// the warp and then across the warps in fp32 with error-free TwoSum pairs.
// Then c = 1/Z, H = ln Z - ln(2) S / Z, u = ln Z - (x_y - m).
//
// Top-k (Section 5.3): a segment's (sequence's) k best eligible rows by (score
// descending, index ascending) on 64-bit keys. Up to 288 rows (one per thread of
// the row kernel's CTA) the last CTA to finish a segment ranks them; it is found
// with a self-resetting counter per segment, incremented with acquire-release
// semantics. Longer segments' lists come from a launch of their own behind the
// rows (topk_kernel), lists of up to 8 rows excepted.
//
// Decision step (cover_score_decide_fwd, Sections 5.2, 3 and 5.3): the row
// pass keeps u of the current token and ln Z (= u of the greedy token) in a
// workspace. Per segment, the most confident masked rows above the threshold
// are then drafted (at most B), Keep / Replace / ReMask applied to the previous
// seeds, the updated state scored, the scores above their mean counted
// (n_t pi_t), and ceil(sqrt(n_t pi_t)) new seeds selected among the rows that
// were not seeds and have ReMasks left, with the same 64-bit keys: by the last
// CTA of a segment up to 288 rows, in a launch of its own (decide_kernel) above.
//
// Streaming: a producer warp issues cp.async.bulk copies of 16 KB chunks of the row's aligned
// 16-byte vectors into a 3-stage shared-memory ring (mbarrier full / empty), 8 consumer warps
// reduce from shared memory; bytes in flight do not cost registers, and 4 CTAs share an SM. The
// up to 14 elements outside the aligned vectors (V or the row's offset not a multiple of 8) are
// read by the producer warp's other lanes. With few rows each is split over the CTAs of a cluster
// (row_split), whose slice sums its first CTA adds. Unaligned rows of which an SM has one or two go
// through a kernel of 16-byte register loads where that is ahead (loads_to_registers); with more
// rows it falls behind: 1024 rows of V = 126465 57.9 against 50.1 us.
#include <math.h>
#include <stdint.h>

#include <algorithm>

#include "cluster.cuh"
#include "context.cuh"
#include "kernels.cuh"
#include "ptx.cuh"

namespace cover {
namespace {

constexpr int kConsumerWarps = 8;          // consumers + 1 producer warp
constexpr int kBulkThreads = (kConsumerWarps + 1) * 32;
constexpr int kChunkElems = 8192;          // 16 KB of bf16 per bulk copy
constexpr int kChunkBytes = kChunkElems * 2;
constexpr int kRingStages = 3;
constexpr int kRegThreads = 512;           // register-load kernel
constexpr int kRegUnroll = 4;
constexpr int kVecPerThread = kChunkElems / 8 / (kConsumerWarps * 32);   // 4
constexpr float kLog2e = 1.4426950408889634f;
constexpr int kMaxPerSeq = 4096;            // rows per segment (the entry points refuse more)
constexpr int kRowLoads = 4;                // rows whose state a thread loads at once (general paths)
constexpr int kRoundsMax = 32;              // selections up to this size by rounds or warp sorts (top_select)
constexpr int kRoundsFew = 8;               // selections up to this size by per-warp rounds (top_rounds)
constexpr int kFusedTopk = kRoundsFew;      // longest list that the row kernel finds in segments longer than its CTAs
constexpr int kMaxWarps = 32;               // the selection kernels run up to 1024 threads
constexpr int kMaxThreads = 32 * kMaxWarps;
constexpr int kRankWarps = 16;              // top_small ranks the published keys of up to this many warps
constexpr int kMaxSplit = 8;                // CTAs a row is split over (the portable cluster size)
constexpr int kMinSlice = 2048;             // elements of a row a CTA gets at least

struct RowAcc {
  float m;     // running maximum logit of this thread's elements
  int mi;      // where m was first reached: the element's index (mu == 0), else the first index of
               // the batch that held it, mu vectors of 8 values a kernel-constant stride apart
  int mu;
  float mref;  // m * log2(e), the exponent reference
  float z, zc; // Kahan sum of 2^t and its compensation
  float s, sc; // Kahan sum of t 2^t and its compensation
};

__device__ __forceinline__ void kahan_add(float& sum, float& c, float x) {
  const float y = x - c;
  const float t = sum + y;
  c = (t - sum) - y;
  sum = t;
}

// t of the maximum itself is the rounding of its reference, up to half a unit in the last place: below
// this reference 2^t can overflow. A masked logit is often the type's lowest value, and it may be the
// maximum of a lane's or a slice's every element: references stop here, where what lies lower has 2^t = 0.
// (A row of nothing else has no finite sums.)
constexpr float kLowestRef = -2147483648.0f;   // -2^31

// Move the exponent reference to a larger maximum new_m.
__device__ __forceinline__ void raise_max(RowAcc& a, float new_m, int new_i, int new_u) {
  const float new_ref = fmaxf(new_m * kLog2e, kLowestRef);
  if (a.m != -INFINITY) {
    const float d = a.mref - new_ref;  // <= 0
    const float f = ex2_approx(d);
    const float z = a.z - a.zc;
    const float s = a.s - a.sc;
    a.s = f * fmaf(d, z, s);
    a.z = f * z;
  }
  a.zc = 0.0f;
  a.sc = 0.0f;
  a.m = new_m;
  a.mi = new_i;
  a.mu = new_u;
  a.mref = new_ref;
}

__device__ __forceinline__ uint4 ld_stream(const uint4* p) {
  uint4 r;
  asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0, %1, %2, %3}, [%4];"
               : "=r"(r.x), "=r"(r.y), "=r"(r.z), "=r"(r.w)
               : "l"(p));
  return r;
}

__device__ __forceinline__ float bf16_to_f32(uint16_t h) { return __uint_as_float(static_cast<uint32_t>(h) << 16); }

__device__ __forceinline__ void acc_scalar(RowAcc& a, float x, int idx) {
  if (x > a.m) raise_max(a, x, idx, 0);
  const float t = fmaf(x, kLog2e, -a.mref);
  const float e = ex2_approx(t);
  kahan_add(a.z, a.zc, e);
  kahan_add(a.s, a.sc, t * e);
}

__device__ __forceinline__ void unpack8(const uint4& w, float (&x)[8]) {
  const uint32_t v[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    x[2 * k] = __uint_as_float(v[k] << 16);
    x[2 * k + 1] = __uint_as_float(v[k] & 0xffff0000u);
  }
}

__device__ __forceinline__ uint32_t order_key(float f) {
  const uint32_t u = __float_as_uint(f);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float order_key_inv(uint32_t k) {
  return __uint_as_float((k & 0x80000000u) ? (k & 0x7fffffffu) : ~k);
}


// ---------------------------------------------------------------------------
// per-row finish (all threads of the CTA call it; NW = warps in the CTA)
// ---------------------------------------------------------------------------
struct RowOut {
  float M;      // row maximum
  int yhat;     // first index attaining it
  float Z;      // sum 2^t re-referenced to M log2(e)
  float q;      // (sum t 2^t) / Z
};

// A row's (or a row slice's) sums as unevaluated pairs (value, rounding error).
struct alignas(8) RowSum {
  float M;        // maximum; -inf for an empty slice
  int yhat;       // first index attaining it
  float zh, zl;   // sum 2^t re-referenced to M log2(e)
  float sh, sl;   // sum t 2^t
};

// a + b = s + e exactly (Knuth's TwoSum)
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
  s = a + b;
  const float bb = s - a;
  e = (a - (s - bb)) + (b - bb);
}

// A thread's recorded batch is re-read, in up to four vectors kStride elements apart, from the ring
// while it still holds the batch's chunk, else from the row in global memory; the loads are issued
// by the threads that hold their warp's maximum before the block-wide maximum is known, so their
// latency overlaps the reduction.
constexpr int kMaxBatch = 4;
static_assert(kVecPerThread <= kMaxBatch && kRegUnroll <= kMaxBatch, "batches hold at most four vectors");

// Where the row kernel's ring holds a row (slice) after its last chunk: element `first` of the row
// began chunk 0, and chunks from `held` on are there.
struct Ring {
  const uint8_t* base;
  int first, held;
};

template <int kStride>
__device__ __forceinline__ void load_batch(const RowAcc& a, const uint16_t* row, const Ring& ring,
                                           uint4 (&w)[kMaxBatch]) {
  const int at = a.mi - ring.first, c = at / kChunkElems;
  const uint16_t* src = a.mu != 0 && c >= ring.held
                            ? reinterpret_cast<const uint16_t*>(ring.base + (c % kRingStages) * kChunkBytes) +
                                  (at - c * kChunkElems)
                            : row + a.mi;
#pragma unroll
  for (int u = 0; u < kMaxBatch; ++u)
    if (u < a.mu) w[u] = *reinterpret_cast<const uint4*>(src + u * kStride);
}

// First index of the value M in the thread's recorded batch w.
template <int kStride>
__device__ __forceinline__ int first_index_of(const RowAcc& a, float M, const uint4 (&w)[kMaxBatch]) {
  if (a.mu == 0) return a.mi;
  int idx = 0x7fffffff;
#pragma unroll
  for (int u = kMaxBatch - 1; u >= 0; --u) {
    if (u >= a.mu) continue;
    float x[8];
    unpack8(w[u], x);
#pragma unroll
    for (int k = 7; k >= 0; --k)
      if (x[k] == M) idx = a.mi + u * kStride + k;
  }
  return idx;
}

template <int NW, int kStride>
__device__ __forceinline__ RowSum row_reduce(const RowAcc& a, const uint16_t* row, const Ring& ring, float* red_m, int* red_i,
                                             float2* red_z, float2* red_s) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  float m = a.m;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  const bool cand = a.m == m && m != -INFINITY;   // may hold the row maximum
  uint4 w[kMaxBatch];
  if (cand) load_batch<kStride>(a, row, ring, w);
  if (lane == 0) red_m[warp] = m;
  __syncthreads();
  float M = red_m[0];
#pragma unroll
  for (int i = 1; i < NW; ++i) M = fmaxf(M, red_m[i]);
  // partials re-referenced to the row maximum (to the unrounded M log2 e), summed across the warp in fp32
  // with error-free TwoSum pairs (value, rounding error), then across the warps
  // the same way by thread 0
  float z = 0.0f, ze = 0.0f, sv = 0.0f, se = 0.0f;
  if (a.m != -INFINITY) {
    const float d = fmaf(-M, kLog2e, a.mref);
    const float f = ex2_approx(d);
    const float zz = a.z - a.zc;
    const float ss = a.s - a.sc;
    z = f * zz;
    sv = f * fmaf(d, zz, ss);
  } else {
    z = a.z - a.zc;   // 0, or NaN if a lane without a maximum has seen one
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const float z2 = __shfl_xor_sync(0xffffffffu, z, o), ze2 = __shfl_xor_sync(0xffffffffu, ze, o);
    const float s2 = __shfl_xor_sync(0xffffffffu, sv, o), se2 = __shfl_xor_sync(0xffffffffu, se, o);
    float t = z + z2, bb = t - z;
    ze += ze2 + ((z - (t - bb)) + (z2 - bb));
    z = t;
    t = sv + s2;
    bb = t - sv;
    se += se2 + ((sv - (t - bb)) + (s2 - bb));
    sv = t;
  }
  // the threads holding the row maximum find its first index in their recorded batches
  const int mi = __reduce_min_sync(0xffffffffu, cand && a.m == M ? first_index_of<kStride>(a, M, w) : 0x7fffffff);
  if (lane == 0) {
    red_i[warp] = mi;
    red_z[warp] = make_float2(z, ze);
    red_s[warp] = make_float2(sv, se);
  }
  __syncthreads();
  RowSum r{M, 0x7fffffff, 0.0f, 0.0f, 0.0f, 0.0f};
  if (tid == 0) {
    int I = red_i[0];
#pragma unroll
    for (int w = 1; w < NW; ++w) I = min(I, red_i[w]);
    r.yhat = I;
    // the warps' (value, error) pairs added with TwoSum in fp32 (no fp64: this GPU's fp64 adds
    // have long latencies, and this runs at the end of every row with no copy in flight)
    r.zh = red_z[0].x, r.zl = red_z[0].y, r.sh = red_s[0].x, r.sl = red_s[0].y;
#pragma unroll
    for (int w = 1; w < NW; ++w) {
      float t, e;
      two_sum(r.zh, red_z[w].x, t, e);
      r.zl += e + red_z[w].y;
      r.zh = t;
      two_sum(r.sh, red_s[w].x, t, e);
      r.sl += e + red_s[w].y;
      r.sh = t;
    }
  }
  return r;
}

// S / Z with one correction step on the pairs: q = sh / zh, then the residual of
// (sh + sl) - q (zh + zl) divided by zh
__device__ __forceinline__ RowOut row_finish(const RowSum& r) {
  const float q0 = r.sh / r.zh;
  const float res = fmaf(-q0, r.zh, r.sh) + (r.sl - q0 * r.zl);
  return {r.M, r.yhat, r.M != -INFINITY ? r.zh + r.zl : 0.0f, q0 + res / r.zh};
}

// The sum of the row slices in part[0 .. C), on the lanes of one warp: every lane returns it.
// Each slice's pairs move to the row maximum (S by the error-free product d zh), then a tree
// of TwoSums adds them, so a split row keeps the accuracy of an unsplit one.
template <int C>
__device__ __forceinline__ RowSum row_combine(const RowSum* part, int lane) {
  RowSum r = part[lane & (C - 1)];
  float M = r.M;
#pragma unroll
  for (int o = C / 2; o > 0; o >>= 1) M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, o));
  int y = r.M == M ? r.yhat : 0x7fffffff;
  if (r.M < M && r.M * kLog2e < kLowestRef) {
    r.zh = r.zl = r.sh = r.sl = 0.0f;   // a slice of masked logits (two such bf16 maxima differ by 2^23 at least)
  } else if (r.M != -INFINITY) {
    // d + dl = (r.M - M) log2 e to twice the precision: its rounding would shift the whole slice
    const float d = __fmul_rn(r.M - M, kLog2e);   // <= 0
    const float dl = fmaf(r.M - M, kLog2e, -d);
    float f = ex2_approx(d);
    f = fmaf(f, 0.6931471805599453f * dl, f);
    const float p = d * r.zh;
    float sh, se;
    two_sum(r.sh, p, sh, se);
    const float sl = se + fmaf(d, r.zh, -p) + fmaf(d, r.zl, r.sl) + dl * r.zh;
    r.sh = f * sh;
    r.sl = fmaf(f, sh, -r.sh) + f * sl;
    const float zh = r.zh;
    r.zh = f * zh;
    r.zl = fmaf(f, zh, -r.zh) + f * r.zl;
  }
#pragma unroll
  for (int o = C / 2; o > 0; o >>= 1) {
    y = min(y, __shfl_xor_sync(0xffffffffu, y, o));
    const float zh2 = __shfl_xor_sync(0xffffffffu, r.zh, o), zl2 = __shfl_xor_sync(0xffffffffu, r.zl, o);
    const float sh2 = __shfl_xor_sync(0xffffffffu, r.sh, o), sl2 = __shfl_xor_sync(0xffffffffu, r.sl, o);
    float t, e;
    two_sum(r.zh, zh2, t, e);
    r.zl += zl2 + e;
    r.zh = t;
    two_sum(r.sh, sh2, t, e);
    r.sl += sl2 + e;
    r.sh = t;
  }
  r.M = M;
  r.yhat = y;
  return r;
}

// What a row's scores need beside its sums, read by the producer while the row streams: the logit of
// the current token y (NaN for a token outside [0, V), which has no probability), d_in and d_out.
// Read after the sums, they were two more round trips to memory at the end of each row: with the
// batches read back from the ring (load_batch) 7.27 -> 6.81 us on 32 rows of 126464 logits with all of
// them given, 19.1 -> 18.4 us on 256 rows, 57.1 -> 55.9 us on 1024 rows of 152064.
// Whether a token is given is a flag of its own: every 32-bit value may come as a token.
struct RowSide {
  bool greedy;   // no current token: y is the row's greedy token
  float xy, din, dout;
};

// The logit of the given current token y; takes the token's load as its latency.
__device__ __forceinline__ void side_logit(RowSide& r, int y, const uint16_t* row, int V) {
  if (r.greedy) return;
  const bool in = y >= 0 && y < V;
  r.xy = in ? bf16_to_f32(row[y]) : __int_as_float(0x7fc00000);
}

// Thread 0 writes the row's outputs; returns (to thread 0) whether this CTA is
// the last of its segment to finish.
__device__ __forceinline__ bool row_write(const RowOut& r, const RowSide& side, int n, int per_seq, int topk,
                                          float* maxprob, float* entropy, int32_t* argmax, float* score,
                                          uint32_t* counters, float* ws_u = nullptr, float* ws_lnz = nullptr) {
  const float Zf = r.Z;
  const float lnZ = logf(Zf);
  const float H = lnZ - 0.6931471805599453f * r.q;
  // a row without a greedy token (no logit above -inf) has no uncertainty of it either
  const float u = !side.greedy ? lnZ - (side.xy - r.M) : r.M != -INFINITY ? lnZ : __int_as_float(0x7fc00000);
  maxprob[n] = 1.0f / Zf;
  entropy[n] = H;
  argmax[n] = r.yhat;
  if (ws_u != nullptr) {
    // decision step: the seed score is formed after the state update
    ws_u[n] = u;
    ws_lnz[n] = lnZ;
    if (counters == nullptr) return false;   // the decisions have a launch of their own
  } else {
    score[n] = u * (1.0f + side.din) / (1.0f + side.dout);
    if (topk <= 0) return false;
  }
  // The counter increment is a release (thread 0 wrote all of the row's results above) and an
  // acquire: the segment's last CTA, after its block barrier, reads the results of the others.
  const unsigned seg = static_cast<unsigned>(n / per_seq);
  unsigned old;
  asm volatile("atom.acq_rel.gpu.global.inc.u32 %0, [%1], %2;"
               : "=r"(old)
               : "l"(counters + seg), "r"(static_cast<unsigned>(per_seq - 1))
               : "memory");
  return old == static_cast<unsigned>(per_seq - 1);
}

constexpr int kDecideFused = 1, kDecideApart = 2;
struct ScoreParams {
  const uint16_t* logits;
  int V, per_seq;
  const int32_t* cur_tok;
  const float* d_in;
  const float* d_out;
  const uint8_t* eligible;
  int topk, sort_n;
  float* maxprob;
  float* entropy;
  int32_t* argmax;
  float* score;
  int32_t* topk_idx;
  float* topk_score;
  uint32_t* counters;
  int decide;          // kDecideFused: the last CTA of a segment decides; kDecideApart: decide_kernel does
  DecideArgs dec;
  bool evict_first;    // see stream_policy
};

// Descending bitonic sort of n (a power of two) 64-bit keys in shared memory;
// all threads of the CTA call it.
__device__ __forceinline__ void bitonic_sort_desc(uint64_t* keys, int n) {
  const int tid = threadIdx.x, nt = blockDim.x;
  for (int k = 2; k <= n; k <<= 1) {
    for (int j = k >> 1; j > 0; j >>= 1) {
      for (int i = tid; i < n; i += nt) {
        const int p = i ^ j;
        if (p > i) {
          const uint64_t x = keys[i], y = keys[p];
          const bool desc = (i & k) == 0;
          if (desc ? (x < y) : (x > y)) {
            keys[i] = y;
            keys[p] = x;
          }
        }
      }
      __syncthreads();
    }
  }
}

// Sum over the CTA (blockDim a multiple of 32); every thread gets the total,
// added in the same order everywhere. scratch: 32 entries.
template <typename T>
__device__ __forceinline__ T block_sum(T v, T* scratch) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  __syncthreads();
  if (lane == 0) scratch[warp] = v;
  __syncthreads();
  T t = 0;
  for (int w = 0; w < nw; ++w) t += scratch[w];
  return t;
}

// A finite fp32 score as a 64-bit fixed-point integer on the binade of the segment's largest
// score (biased exponent emax): s 2^(26 - E), |result| < 2^50. Exact for a score within a factor
// 2^26 of the largest; a smaller one is truncated toward zero. Sums of up to 4096 of them and
// their products with counts up to 4096 stay below 2^62, so the mean test n_t s > sum s is an
// exact integer comparison on these values.
__device__ __forceinline__ long long fixed_of(float s, uint32_t emax) {
  const uint32_t bits = __float_as_uint(s);
  const uint32_t eb = (bits >> 23) & 0xffu;
  // s = m 2^(eb - 150) (m with its leading bit; a denormal has eb 0 and exponent 1 - 150)
  const uint32_t m = eb != 0u ? ((bits & 0x7fffffu) | 0x800000u) : (bits & 0x7fffffu);
  const int shift = static_cast<int>(eb == 0u ? 1u : eb) - static_cast<int>(emax) + 26;
  const long long mag = shift >= 0 ? (static_cast<long long>(m) << shift) : (shift > -25 ? (m >> -shift) : 0);
  return (bits >> 31) ? -mag : mag;
}

// key of row i ordered by value descending, then index ascending; 0 = no row
__device__ __forceinline__ uint64_t rank_key(float v, int i) {
  return (static_cast<uint64_t>(order_key(v)) << 32) | (0xffffffffu - static_cast<uint32_t>(i));
}
__device__ __forceinline__ int rank_key_row(uint64_t key) {
  return static_cast<int>(0xffffffffu - static_cast<uint32_t>(key));
}

// Descending bitonic sorts of G independent sets of 32 keys across the warp (key[g]: lane t's
// key of set g), by shuffles; the G sets go through the network together.
template <int G>
__device__ __forceinline__ void warp_sort_desc(uint64_t (&key)[G], int lane) {
#pragma unroll
  for (int size = 2; size <= 32; size <<= 1) {
    const bool desc = (lane & size) == 0;
#pragma unroll
    for (int stride = size >> 1; stride > 0; stride >>= 1) {
      const bool take_max = ((lane & stride) == 0) == desc;
#pragma unroll
      for (int g = 0; g < G; ++g) {
        const uint64_t other = __shfl_xor_sync(0xffffffffu, key[g], stride);
        key[g] = take_max ? (key[g] > other ? key[g] : other) : (key[g] < other ? key[g] : other);
      }
    }
  }
}
__device__ __forceinline__ uint64_t warp_sort_desc(uint64_t key, int lane) {
  uint64_t k1[1] = {key};
  warp_sort_desc<1>(k1, lane);
  return k1[0];
}

// a[g] becomes the 32 largest of the descending lists a[g] and b[g] (lane t holds the t-th of
// each), descending: the larger of a[t] and b[31 - t] is a bitonic sequence holding them, which
// the half-cleaners of strides 16 .. 1 put in order. The G merges go through together.
template <int G>
__device__ __forceinline__ void warp_merge_desc(uint64_t (&a)[G], const uint64_t (&b)[G], int lane) {
#pragma unroll
  for (int g = 0; g < G; ++g) {
    const uint64_t br = __shfl_sync(0xffffffffu, b[g], 31 - lane);
    a[g] = a[g] > br ? a[g] : br;
  }
#pragma unroll
  for (int stride = 16; stride > 0; stride >>= 1) {
    const bool take_max = (lane & stride) == 0;
#pragma unroll
    for (int g = 0; g < G; ++g) {
      const uint64_t other = __shfl_xor_sync(0xffffffffu, a[g], stride);
      a[g] = take_max ? (a[g] > other ? a[g] : other) : (a[g] < other ? a[g] : other);
    }
  }
}

// Number of entries of the descending list l[0 .. 32) larger than x (x not in the list).
__device__ __forceinline__ int count_above(const uint64_t* l, uint64_t x) {
  int c = 0;
#pragma unroll
  for (int step = 32; step > 0; step >>= 1)
    if (c + step <= 32 && l[c + step - 1] > x) c += step;
  return c;
}

// Largest of the warp's 64-bit values (two 32-bit reductions: the high words, then the low
// words of the lanes that hold the largest high word).
__device__ __forceinline__ uint64_t warp_max_u64(uint64_t x) {
  const uint32_t hi = __reduce_max_sync(0xffffffffu, static_cast<uint32_t>(x >> 32));
  const uint32_t lo = __reduce_max_sync(0xffffffffu, static_cast<uint32_t>(x >> 32) == hi ? static_cast<uint32_t>(x) : 0u);
  return (static_cast<uint64_t>(hi) << 32) | lo;
}

// The k largest (k <= kRoundsFew) of the n keys in shared memory (keys are distinct, 0 = none),
// in descending order: out[t] gets the t-th (0 once the nonzero keys run out). Each warp takes
// its own k largest by k rounds of a warp-wide maximum below the previous round's (no block
// barrier per round), over the keys its lanes read (i = tid, tid + blockDim, ...); a key can be
// among the k largest only if it is among its warp's, so ranking the warps' lists against each
// other is exact below k. All threads call it with the same k.
__device__ __forceinline__ void top_rounds(const uint64_t* keys, int n, int k, uint64_t* out) {
  __shared__ uint64_t s_list[kMaxWarps * kRoundsFew];
  const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, warp = tid >> 5, nw = nt >> 5;
  if (k <= 0) return;
  uint64_t prev = ~0ull;
  for (int t = 0; t < k; ++t) {
    uint64_t m = 0;
    for (int i = tid; i < n; i += nt) {
      const uint64_t x = keys[i];
      if (x < prev && x > m) m = x;
    }
    prev = warp_max_u64(m);
    if (lane == 0) s_list[warp * k + t] = prev;   // 0 once the warp's keys run out
  }
  const int nl = nw * k;
  __syncthreads();
  const uint64_t key = tid < nl ? s_list[tid] : 0;
  const int listed = __syncthreads_count(key != 0);
  if (key != 0) {
    int r = 0;
    for (int j = 0; j < nl; ++j) r += s_list[j] > key ? 1 : 0;
    if (r < k) out[r] = key;
  }
  for (int t = min(listed, k) + tid; t < k; t += nt) out[t] = 0;
  __syncthreads();
}

// The k largest (k <= 32) of the n keys in shared memory (distinct, 0 = none), in descending
// order: out[t] gets the t-th (0 once the nonzero keys run out). Each warp keeps the 32 largest
// keys it has read in registers (lane t: the t-th). It reads four sets of 32 keys at a time
// (every (warps)-th set of the array), sorts them together, merges them pairwise and folds the
// result into its list, skipping the work when no key passes the list's k-th. A key can be
// among the k largest only if it is among its warp's, so the warps' lists decide the result:
// a listed key's rank is its position in its own list plus the number of larger keys in each
// other list (a binary search, the lists being sorted), exact below k. The lists are staged in
// keys[0 .. 32 * warps), which n >= blockDim.x guarantees; the keys are not read afterwards.
// All threads call it with the same k.
__device__ __forceinline__ void top_warps(uint64_t* keys, int n, int k, uint64_t* out) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = blockDim.x >> 5;
  if (k <= 0) return;
  constexpr int kSets = 4;
  uint64_t top[1] = {0};
  for (int j0 = warp * 32 + lane; j0 - lane < n; j0 += kSets * nw * 32) {
    uint64_t b[kSets];
#pragma unroll
    for (int g = 0; g < kSets; ++g) {
      const int j = j0 + g * nw * 32;
      b[g] = j < n ? keys[j] : 0;
    }
    const uint64_t kth = __shfl_sync(0xffffffffu, top[0], k - 1);
    if (!__any_sync(0xffffffffu, b[0] > kth || b[1] > kth || b[2] > kth || b[3] > kth)) continue;
    warp_sort_desc<kSets>(b, lane);
    uint64_t p[2] = {b[0], b[2]};
    const uint64_t q[2] = {b[1], b[3]};
    warp_merge_desc<2>(p, q, lane);
    const uint64_t p1[1] = {p[1]};
    uint64_t p0[1] = {p[0]};
    warp_merge_desc<1>(p0, p1, lane);
    warp_merge_desc<1>(top, p0, lane);
  }
  __syncthreads();   // every warp is done reading the keys
  keys[warp * 32 + lane] = lane < k ? top[0] : 0;
  const int published = __syncthreads_count(lane < k && top[0] != 0);
  if (lane < k && top[0] != 0) {
    int r = lane;
#pragma unroll 4
    for (int w = 0; w < nw; ++w)
      if (w != warp) r += count_above(keys + w * 32, top[0]);
    if (r < k) out[r] = top[0];
  }
  for (int t = min(published, k) + tid; t < k; t += blockDim.x) out[t] = 0;
  __syncthreads();
}

// The k largest (k <= kRoundsMax) of n keys in shared memory into out, by rounds for a few keys
// and by warp sorts otherwise; the first 32 * warps keys may be overwritten.
__device__ __forceinline__ void top_select(uint64_t* keys, int n, int k, uint64_t* out) {
  if (k <= kRoundsFew)
    top_rounds(keys, n, k, out);
  else
    top_warps(keys, n, k, out);
}

// Sections 5.2 and 3 for a segment of any length, by one CTA: drafting and the
// revision of the previous seeds. Updates tok, remask_cnt, flags (bit 1 marks
// the rows drafted in this step; a drafted row loses bit 0) and ws_u (the
// uncertainty of each row's updated token: ln Z for drafted and replaced rows).
// Rows written by other CTAs are read through L2 (__ldcg). The drafting sort
// runs only when more rows pass the threshold than the budget allows.
__device__ void segment_update(uint64_t* keys, int seg, int per_seq, int sort_n, const ScoreParams& P) {
  __shared__ unsigned long long s_fallback;
  __shared__ uint32_t s_draft_bits[kMaxPerSeq / 32];
  __shared__ int s_ri[32];
  __shared__ int s_cnt[3][32];
  __shared__ uint64_t s_sel[kRoundsMax];
  const DecideArgs& d = P.dec;
  const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, warp = tid >> 5, nw = nt >> 5;
  const int base = seg * per_seq;
  if (tid == 0) s_fallback = ~0ull;
  __syncthreads();

  // Section 5.2 drafting: masked rows in the allowed set whose confidence exceeds tau. Each
  // thread loads the state of kRowLoads rows before it uses any of it (the loads of a batch
  // overlap instead of waiting on one another's results).
  int ncand = 0;
  uint64_t fb_min = ~0ull;   // the thread's lowest (entropy, index) key among allowed rows
  for (int i0 = tid; i0 < per_seq; i0 += kRowLoads * nt) {
    bool allowed[kRowLoads];
    float c[kRowLoads], h[kRowLoads];
#pragma unroll
    for (int u = 0; u < kRowLoads; ++u) {
      const int i = i0 + u * nt;
      const bool in = i < per_seq;
      const int n = base + (in ? i : 0);
      allowed[u] = in && d.tok[n] == d.mask_id & (d.draft_ok == nullptr || d.draft_ok[n] != 0);
      c[u] = __ldcg(P.maxprob + n);
      h[u] = __ldcg(P.entropy + n);
    }
#pragma unroll
    for (int u = 0; u < kRowLoads; ++u) {
      if (!allowed[u]) continue;
      if (c[u] > d.tau) ++ncand;
      // lowest entropy, then lowest index
      const uint64_t fb = (static_cast<uint64_t>(order_key(h[u])) << 32) | static_cast<uint32_t>(i0 + u * nt);
      fb_min = fb < fb_min ? fb : fb_min;
    }
  }
  if (d.min_one) {
    // one shared-memory atomic per warp (a 64-bit minimum by two 32-bit reductions)
    const uint32_t hi = __reduce_min_sync(0xffffffffu, static_cast<uint32_t>(fb_min >> 32));
    const uint32_t lo =
        __reduce_min_sync(0xffffffffu, static_cast<uint32_t>(fb_min >> 32) == hi ? static_cast<uint32_t>(fb_min) : ~0u);
    const uint64_t wmin = (static_cast<uint64_t>(hi) << 32) | lo;   // ~0 only when no lane has a row
    if (lane == 0 && wmin != ~0ull) atomicMin(&s_fallback, static_cast<unsigned long long>(wmin));
  }
  ncand = block_sum(ncand, s_ri);
  const bool all_cand = ncand <= d.budget;   // every row above tau is drafted
  int n_drafted = min(ncand, d.budget);
  const bool fallback = n_drafted == 0 && d.min_one && s_fallback != ~0ull;
  if (!all_cand) {
    // more candidates than the budget: the `budget` most confident (ties to the lower index)
    for (int i0 = tid; i0 < sort_n; i0 += kRowLoads * nt) {
      bool allowed[kRowLoads];
      float c[kRowLoads];
#pragma unroll
      for (int u = 0; u < kRowLoads; ++u) {
        const int i = i0 + u * nt;
        const bool in = i < per_seq;
        const int n = base + (in ? i : 0);
        allowed[u] = in && d.tok[n] == d.mask_id & (d.draft_ok == nullptr || d.draft_ok[n] != 0);
        c[u] = __ldcg(P.maxprob + n);
      }
#pragma unroll
      for (int u = 0; u < kRowLoads; ++u) {
        const int i = i0 + u * nt;
        if (i < sort_n) keys[i] = allowed[u] && c[u] > d.tau ? rank_key(c[u], i) : 0;
      }
    }
    __syncthreads();
    if (n_drafted <= kRoundsMax)
      top_select(keys, sort_n, n_drafted, s_sel);
    else
      bitonic_sort_desc(keys, sort_n);
  }
  // the drafted rows, marked for the pass below when they were selected (more candidates than
  // the budget) or are the fallback row; with every candidate drafted the pass decides itself
  if (!all_cand || fallback) {
    for (int w = tid; w < kMaxPerSeq / 32; w += nt) s_draft_bits[w] = 0u;
    __syncthreads();
    const uint64_t* picked = n_drafted <= kRoundsMax ? s_sel : keys;
    for (int t = tid; t < (fallback ? 1 : n_drafted); t += nt) {
      const int i = fallback ? static_cast<int>(static_cast<uint32_t>(s_fallback)) : rank_key_row(picked[t]);
      atomicOr(&s_draft_bits[i >> 5], 1u << (i & 31));
    }
    __syncthreads();
  }
  const bool marked = !all_cand || fallback;
  if (fallback) n_drafted = 1;

  // Section 5.2 revision of the previous seeds, Section 3 state update
  int kept = 0, replaced = 0, remasked = 0;
  for (int i0 = tid; i0 < per_seq; i0 += kRowLoads * nt) {
    int y[kRowLoads], yh[kRowLoads];
    uint32_t fl[kRowLoads], rc[kRowLoads];
    bool ok[kRowLoads];
    float c[kRowLoads], lz[kRowLoads];
#pragma unroll
    for (int u = 0; u < kRowLoads; ++u) {
      const int i = i0 + u * nt;
      const int n = base + (i < per_seq ? i : 0);
      y[u] = d.tok[n];
      fl[u] = d.flags[n];
      rc[u] = d.remask_cnt[n];
      ok[u] = d.draft_ok == nullptr || d.draft_ok[n] != 0;
      c[u] = __ldcg(P.maxprob + n);
      yh[u] = __ldcg(P.argmax + n);
      lz[u] = __ldcg(d.ws_lnz + n);
    }
#pragma unroll
    for (int u = 0; u < kRowLoads; ++u) {
      const int i = i0 + u * nt;
      if (i >= per_seq) continue;
      const int n = base + i;
      const bool drafted = marked ? (s_draft_bits[i >> 5] >> (i & 31)) & 1u
                                  : y[u] == d.mask_id && ok[u] && c[u] > d.tau;
      if (drafted) {
        // a drafted row takes its greedy token, whose uncertainty is ln Z
        d.tok[n] = yh[u];
        d.ws_u[n] = lz[u];
        d.flags[n] = static_cast<uint8_t>((fl[u] & ~1u) | 2u);
      } else if ((fl[u] & 1u) != 0 && y[u] != d.mask_id) {
        if (yh[u] == y[u]) {
          ++kept;
        } else if (c[u] > d.tau) {
          ++replaced;
          d.tok[n] = yh[u];
          d.ws_u[n] = lz[u];
        } else {
          ++remasked;
          d.tok[n] = d.mask_id;
          d.remask_cnt[n] = static_cast<uint8_t>(min(rc[u] + 1u, 255u));
        }
      }
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    kept += __shfl_xor_sync(0xffffffffu, kept, o);
    replaced += __shfl_xor_sync(0xffffffffu, replaced, o);
    remasked += __shfl_xor_sync(0xffffffffu, remasked, o);
  }
  if (lane == 0) {
    s_cnt[0][warp] = kept;
    s_cnt[1][warp] = replaced;
    s_cnt[2][warp] = remasked;
  }
  __syncthreads();
  if (tid == 0 && d.stats != nullptr) {
    kept = replaced = remasked = 0;
    for (int w = 0; w < nw; ++w) {
      kept += s_cnt[0][w];
      replaced += s_cnt[1][w];
      remasked += s_cnt[2][w];
    }
    int32_t* st = d.stats + static_cast<size_t>(seg) * kDecideStats;
    st[0] = n_drafted;
    st[1] = kept;
    st[2] = replaced;
    st[3] = remasked;
  }
}

// Section 5.3 on the updated state of one segment (all threads of the CTA):
// seed score of every unmasked row, the adaptive revision rate, and the
// selection among rows that were not previous seeds and have ReMasks left.
// Clears flag bits 0 and 1 everywhere, then sets bit 0 on the new seeds.
// keys: sort_n 64-bit slots of shared memory followed by sort_n floats.
__device__ void segment_select(uint64_t* keys, int seg, int per_seq, int sort_n, const DecideArgs& d,
                               const float* d_in, const float* d_out, float* score) {
  __shared__ int s_ri[32];
  __shared__ int s_nt[32];
  __shared__ uint32_t s_em[32];
  __shared__ long long s_fx[32];
  __shared__ uint64_t s_sel[kRoundsMax];
  const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, warp = tid >> 5, nw = nt >> 5;
  const int base = seg * per_seq;
  float* sscore = reinterpret_cast<float*>(keys + sort_n);   // per-row seed score

  int n_t = 0;
  uint32_t emax = 0;   // largest biased exponent of the finite scores
  for (int i0 = tid; i0 < sort_n; i0 += kRowLoads * nt) {
    // the state of kRowLoads rows, loaded before any of it is used
    uint32_t fl[kRowLoads], rc[kRowLoads];
    int tk[kRowLoads];
    float din[kRowLoads], dout[kRowLoads], uu[kRowLoads];
#pragma unroll
    for (int u = 0; u < kRowLoads; ++u) {
      const int i = i0 + u * nt;
      const int n = base + (i < per_seq ? i : 0);
      fl[u] = d.flags[n];
      rc[u] = d.remask_cnt[n];
      tk[u] = d.tok[n];
      din[u] = d_in != nullptr ? d_in[n] : 0.0f;
      dout[u] = d_out != nullptr ? d_out[n] : 0.0f;
      uu[u] = __ldcg(d.ws_u + n);
    }
#pragma unroll
    for (int u = 0; u < kRowLoads; ++u) {
      const int i = i0 + u * nt;
      if (i >= sort_n) continue;
      uint64_t key = 0;
      if (i < per_seq) {
        const int n = base + i;
        float s = -INFINITY;
        if (tk[u] != d.mask_id) {
          const float sc = uu[u] * (1.0f + din[u]) / (1.0f + dout[u]);
          if (isfinite(sc)) {
            s = sc;
            ++n_t;
            emax = max(emax, (__float_as_uint(sc) >> 23) & 0xffu);
            if ((fl[u] & 1u) == 0 && static_cast<int>(rc[u]) < d.remask_budget) key = rank_key(sc, i);
          }
        }
        score[n] = s;
        sscore[i] = s;
        d.flags[n] = static_cast<uint8_t>(fl[u] & ~3u);
      }
      keys[i] = key;
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) n_t += __shfl_xor_sync(0xffffffffu, n_t, o);
  emax = __reduce_max_sync(0xffffffffu, emax);
  if (lane == 0) {
    s_nt[warp] = n_t;
    s_em[warp] = emax;
  }
  __syncthreads();
  n_t = 0;
  emax = 0;
  for (int w = 0; w < nw; ++w) {
    n_t += s_nt[w];
    emax = max(emax, s_em[w]);
  }
  // the sum of the scores, exact in fixed point (fixed_of)
  long long part = 0;
  for (int i = tid; i < per_seq; i += nt) {
    const float s = sscore[i];
    if (s != -INFINITY) part += fixed_of(s, emax);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
  if (lane == 0) s_fx[warp] = part;
  __syncthreads();
  long long total = 0;
  for (int w = 0; w < nw; ++w) total += s_fx[w];

  // adaptive revision rate: n_t pi_t = #{ s_j > mean } = #{ n_t s_j > sum s }
  int above = 0;
  for (int i = tid; i < per_seq; i += nt) {
    const float s = sscore[i];
    if (s != -INFINITY && static_cast<long long>(n_t) * fixed_of(s, emax) > total) ++above;
  }
  above = block_sum(above, s_ri);
  int k = 0;
  while (k * k < above) ++k;   // ceil(sqrt(n_t pi_t))
  k = min(k, d.max_seeds);

  // the k best eligible rows (keys written above)
  const uint64_t* best = keys;
  if (k > 0 && k <= kRoundsMax) {
    top_select(keys, sort_n, k, s_sel);
    best = s_sel;
  } else if (k > 0) {
    bitonic_sort_desc(keys, sort_n);
  }
  int chosen = 0;
  for (int t = tid; t < d.max_seeds; t += nt) {
    int pos = -1;
    if (t < k && t < sort_n && best[t] != 0) {
      const int i = rank_key_row(best[t]);
      pos = d.pos0 + i;
      d.flags[base + i] = static_cast<uint8_t>(d.flags[base + i] | 1u);
      ++chosen;
    }
    d.seed_idx[static_cast<size_t>(seg) * d.max_seeds + t] = pos;
  }
  chosen = block_sum(chosen, s_ri);
  if (tid == 0) {
    d.n_seeds[seg] = chosen;
    if (d.stats != nullptr) {
      int32_t* st = d.stats + static_cast<size_t>(seg) * kDecideStats;
      st[4] = n_t;
      st[5] = above;
    }
  }
}

// ---------------------------------------------------------------------------
// Fast path of the per-segment work when the segment has at most one row per
// thread of the CTA (per_seq <= blockDim.x): row i belongs to thread i, which
// loads the row's state once (independent loads, one round trip to L2), keeps
// it in registers and writes it back once. Each count takes one barrier
// (__syncthreads_count). A top selection ranks every candidate against the
// other candidates' keys in shared memory: its rank is the number of larger
// keys, so the row of rank r < k is the (r+1)-th best and fills slot r. Keys
// embed the row index, so they are distinct and the result is the general
// path's (the sort or the warp sorts) exactly.
// ---------------------------------------------------------------------------

// Rank of x among keys[0 .. n) (16-byte aligned): the number of larger keys, counted only while
// it can still be below k. All threads read the same entries at the same time (shared-memory
// broadcasts, two keys per load); a warp stops once every lane's count has reached k (x = 0,
// no key, counts as already there), and the result is then some value >= k.
__device__ __forceinline__ int rank_below(const uint64_t* keys, int n, uint64_t x, int k) {
  int r = x != 0 ? 0 : k;
  const ulonglong2* k2 = reinterpret_cast<const ulonglong2*>(keys);
  int j = 0;
  for (; j + 32 <= n; j += 32) {
    if (__all_sync(0xffffffffu, r >= k)) return r;
#pragma unroll
    for (int q = 0; q < 16; ++q) {
      const ulonglong2 y = k2[(j >> 1) + q];
      r += (y.x > x ? 1 : 0) + (y.y > x ? 1 : 0);
    }
  }
  for (; j < n; ++j) r += keys[j] > x ? 1 : 0;
  return r;
}


// The 32 largest of the CTA's keys, descending, on the lanes of warp 0: the warps' sorted lists merged
// pairwise (log2(warps) barriers). `sorted` is this lane's key of its warp's list; the merged list of the
// last merge a warp took part in is returned. All threads of the CTA call it; cand holds blockDim.x keys.
__device__ __forceinline__ uint64_t top_merged(uint64_t sorted, uint64_t* cand) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  cand[threadIdx.x] = sorted;
  for (int n = blockDim.x >> 5; n > 1;) {
    // the upper half's lists go into the lower half's
    const int half = (n + 1) >> 1;
    __syncthreads();
    if (warp + half < n) {
      uint64_t mine[1] = {sorted};
      const uint64_t other[1] = {cand[(warp + half) * 32 + lane]};
      warp_merge_desc<1>(mine, other, lane);
      sorted = mine[0];
      cand[threadIdx.x] = sorted;
    }
    n = half;
  }
  return sorted;
}

// The k largest (k <= 32) of the CTA's keys, one per thread (distinct, 0 = none). Each warp sorts
// its keys and publishes its k largest in cand[warp * k ..]; a key can be among the CTA's k
// largest only if it is among its warp's, and the number of larger published keys is its rank,
// exact while below k (a warp publishes at most k). With many warps the
// sorted lists are merged instead, since ranking against every published key would cost warps * k
// reads a thread. Returns, for the key this lane then holds
// (*held), its slot 0 .. k-1 among the CTA's k largest, else -1. All threads of the CTA call it;
// cand holds blockDim.x keys.
// kMerge: the CTA may have more than kRankWarps warps.
template <bool kMerge>
__device__ __forceinline__ int top_small(uint64_t key, int k, uint64_t* cand, uint64_t* held) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  uint64_t sorted = warp_sort_desc(key, lane);
  if (kMerge && nw > kRankWarps) {
    *held = sorted = top_merged(sorted, cand);
    return warp == 0 && lane < k && sorted != 0 ? lane : -1;
  }
  if (lane < k) cand[warp * k + lane] = sorted;
  __syncthreads();
  int slot = -1;
  if (lane < k && sorted != 0) {
    int r = 0;
    for (int j = 0; j < nw * k; ++j) r += cand[j] > sorted ? 1 : 0;
    if (r < k) slot = r;
  }
  *held = sorted;
  return slot;
}

// Section 5.3 on the updated state, one row per thread (see segment_select for the
// general path): seed score, n_t and the mean, n_t pi_t = #{n_t s_j > sum s}, and
// the selection of ceil(sqrt(n_t pi_t)) rows by rank. Writes score, flags and the
// segment's seed list, count and stats[4..5].
template <bool kMerge>
__device__ void select_fast(uint64_t* keys, int seg, int per_seq, const DecideArgs& d, bool in, int tok,
                            uint32_t& fl, uint32_t rc, float u, float din, float dout, float* score) {
  __shared__ long long s_fx[32];
  __shared__ uint32_t s_emax;
  __shared__ int s_elig;
  __shared__ uint8_t s_mark[kMaxThreads];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = blockDim.x >> 5;
  const int n = seg * per_seq + tid;
  float sc = -INFINITY;
  bool valid = false;
  uint64_t key = 0;
  if (in && tok != d.mask_id) {
    const float v = u * (1.0f + din) / (1.0f + dout);
    if (isfinite(v)) {
      sc = v;
      valid = true;
      if ((fl & 1u) == 0 && static_cast<int>(rc) < d.remask_budget) key = rank_key(v, tid);
    }
  }
  // n_t pi_t = #{n_t s_j > sum s} in exact integer arithmetic on the scores' fixed-point values
  // (fixed_of); a score too small to be exact lies far below the mean, and the sum's error
  // stays below n_t units, 2^-50 of the largest score. This GPU's fp64 units have long
  // latencies, so no fp64 is used here.
  const uint32_t sbits = __float_as_uint(sc);
  const uint32_t ebias = valid ? ((sbits >> 23) & 0xffu) : 0u;
  const uint32_t emax_w = __reduce_max_sync(0xffffffffu, ebias);
  const uint32_t eb = __ballot_sync(0xffffffffu, key != 0);
  if (tid == 0) {
    s_elig = 0;
    s_emax = 0u;
  }
  if (in) keys[tid] = key;
  __syncthreads();
  if (lane == 0) {
    atomicMax(&s_emax, emax_w);
    if (eb != 0u) atomicAdd(&s_elig, __popc(eb));
  }
  const int n_t = __syncthreads_count(valid);
  const long long fx = valid ? fixed_of(sc, s_emax) : 0;
  long long tot = fx;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) tot += __shfl_xor_sync(0xffffffffu, tot, o);
  if (lane == 0) s_fx[warp] = tot;
  __syncthreads();
  long long total = 0;
  for (int w = 0; w < nw; ++w) total += s_fx[w];
  const bool is_above = valid && static_cast<long long>(n_t) * fx > total;
  const int above = __syncthreads_count(is_above);
  int k = 0;
  while (k * k < above) ++k;   // ceil(sqrt(n_t pi_t))
  k = min(k, d.max_seeds);
  const int chosen = min(k, s_elig);
  bool chosen_row = false;
  if (k > 0 && k <= 32) {
    // few seeds: per-warp sorts and the ranks of the published keys; the lane holding a chosen
    // key writes its slot and marks the row for its owner thread
    uint64_t held;
    if (in) s_mark[tid] = 0;
    const int slot = top_small<kMerge>(key, k, keys, &held);
    if (slot >= 0) {
      const int row = rank_key_row(held);
      d.seed_idx[static_cast<size_t>(seg) * d.max_seeds + slot] = d.pos0 + row;
      s_mark[row] = 1;
    }
    __syncthreads();
    chosen_row = in && s_mark[tid] != 0;
  } else if (k > 0) {
    const int r = rank_below(keys, per_seq, key, k);
    if (key != 0 && r < k) {
      chosen_row = true;
      d.seed_idx[static_cast<size_t>(seg) * d.max_seeds + r] = d.pos0 + tid;
    }
  }
  if (in) {
    score[n] = sc;
    fl = (fl & ~3u) | (chosen_row ? 1u : 0u);
  }
  for (int t = chosen + tid; t < d.max_seeds; t += blockDim.x) d.seed_idx[static_cast<size_t>(seg) * d.max_seeds + t] = -1;
  if (tid == 0) {
    d.n_seeds[seg] = chosen;
    if (d.stats != nullptr) {
      int32_t* st = d.stats + static_cast<size_t>(seg) * kDecideStats;
      st[4] = n_t;
      st[5] = above;
    }
  }
}

// One segment's decision step, one row per thread (see segment_update and
// segment_select for the general path).
template <bool kMerge>
__device__ void decide_fast(uint64_t* keys, int seg, int per_seq, const ScoreParams& P) {
  __shared__ unsigned long long s_fallback;
  __shared__ int s_cnt[3];
  __shared__ uint8_t s_draft[kMaxThreads];
  const DecideArgs& d = P.dec;
  const int tid = threadIdx.x, lane = tid & 31;
  const bool in = tid < per_seq;
  const int n = seg * per_seq + tid;
  const bool select = d.phase == 0;
  // the row's whole state, in one round trip (other CTAs' results through L2)
  int tok = 0, yhat = 0;
  uint32_t fl = 0, rc = 0;
  float c = 0.0f, H = 0.0f, u = 0.0f, lnz = 0.0f, din = 0.0f, dout = 0.0f;
  bool ok_draft = false;
  if (in) {
    tok = d.tok[n];
    fl = d.flags[n];
    rc = d.remask_cnt[n];
    ok_draft = d.draft_ok == nullptr || d.draft_ok[n] != 0;
    c = __ldcg(P.maxprob + n);
    H = __ldcg(P.entropy + n);
    yhat = __ldcg(P.argmax + n);
    u = __ldcg(d.ws_u + n);
    lnz = __ldcg(d.ws_lnz + n);
    if (select) {
      din = P.d_in != nullptr ? P.d_in[n] : 0.0f;
      dout = P.d_out != nullptr ? P.d_out[n] : 0.0f;
    }
  }
  if (tid == 0) {
    s_fallback = ~0ull;
    s_cnt[0] = s_cnt[1] = s_cnt[2] = 0;
  }
  __syncthreads();

  // Section 5.2 drafting: masked rows in the allowed set whose confidence exceeds tau
  const bool allowed = in && tok == d.mask_id && ok_draft;
  const bool cand = allowed && c > d.tau;
  if (d.min_one) {
    // lowest entropy, then lowest index: a warp minimum (two 32-bit reductions), then one
    // shared-memory atomic per warp
    const uint64_t fb = allowed ? (static_cast<uint64_t>(order_key(H)) << 32) | static_cast<uint32_t>(tid) : ~0ull;
    const uint32_t hi = __reduce_min_sync(0xffffffffu, static_cast<uint32_t>(fb >> 32));
    const uint32_t lo =
        __reduce_min_sync(0xffffffffu, static_cast<uint32_t>(fb >> 32) == hi ? static_cast<uint32_t>(fb) : ~0u);
    const uint64_t wmin = (static_cast<uint64_t>(hi) << 32) | lo;   // ~0 only when no lane has a row
    if (lane == 0 && wmin != ~0ull) atomicMin(&s_fallback, static_cast<unsigned long long>(wmin));
  }
  const int ncand = __syncthreads_count(cand);
  const bool all_cand = ncand <= d.budget;   // every row above tau is drafted
  int n_drafted = min(ncand, d.budget);
  bool drafted = all_cand && cand;
  if (!all_cand) {
    // more candidates than the budget: the `budget` most confident (ties to the lower index)
    const uint64_t ck = cand ? rank_key(c, tid) : 0ull;
    if (d.budget <= 32) {
      if (in) s_draft[tid] = 0;
      uint64_t held;
      const int slot = top_small<kMerge>(ck, d.budget, keys, &held);
      if (slot >= 0) s_draft[rank_key_row(held)] = 1;
      __syncthreads();
      drafted = in && s_draft[tid] != 0;
    } else {
      if (in) keys[tid] = ck;
      __syncthreads();
      drafted = rank_below(keys, per_seq, ck, d.budget) < d.budget && cand;
    }
    __syncthreads();   // the keys are rewritten by the selection
  }
  if (n_drafted == 0 && d.min_one && s_fallback != ~0ull) {
    n_drafted = 1;
    drafted = in && tid == static_cast<int>(static_cast<uint32_t>(s_fallback));
  }

  // Section 5.2 revision of the previous seeds, Section 3 state update
  bool kept = false, replaced = false, remasked = false;
  if (drafted) {
    // a drafted row takes its greedy token, whose uncertainty is ln Z
    tok = yhat;
    u = lnz;
    fl = (fl & ~1u) | 2u;
  } else if (in && (fl & 1u) != 0 && tok != d.mask_id) {
    if (yhat == tok) {
      kept = true;
    } else if (c > d.tau) {
      replaced = true;
      tok = yhat;
      u = lnz;
    } else {
      remasked = true;
      tok = d.mask_id;
      rc = min(rc + 1u, 255u);
    }
  }
  const uint32_t bk = __ballot_sync(0xffffffffu, kept), br = __ballot_sync(0xffffffffu, replaced),
                 bm = __ballot_sync(0xffffffffu, remasked);
  if (lane == 0) {
    if (bk) atomicAdd(&s_cnt[0], __popc(bk));
    if (br) atomicAdd(&s_cnt[1], __popc(br));
    if (bm) atomicAdd(&s_cnt[2], __popc(bm));
  }
  if (select) select_fast<kMerge>(keys, seg, per_seq, d, in, tok, fl, rc, u, din, dout, P.score);
  else __syncthreads();
  if (in) {
    d.tok[n] = tok;
    d.flags[n] = static_cast<uint8_t>(fl);
    d.remask_cnt[n] = static_cast<uint8_t>(rc);
    d.ws_u[n] = u;
  }
  if (tid == 0 && d.stats != nullptr) {
    int32_t* st = d.stats + static_cast<size_t>(seg) * kDecideStats;
    st[0] = n_drafted;
    st[1] = s_cnt[0];
    st[2] = s_cnt[1];
    st[3] = s_cnt[2];
  }
}

// A segment of any length: the update, then (unless only the update was asked
// for) the selection with the caller's d_in / d_out.
__device__ void segment_decide(uint64_t* keys, int seg, int per_seq, int sort_n, const ScoreParams& P) {
  if (per_seq <= static_cast<int>(blockDim.x)) {
    decide_fast<true>(keys, seg, per_seq, P);
    return;
  }
  segment_update(keys, seg, per_seq, sort_n, P);
  if (P.dec.phase == 0) {
    __syncthreads();
    segment_select(keys, seg, per_seq, sort_n, P.dec, P.d_in, P.d_out, P.score);
  }
}

// Top-k of a segment by (score desc, index asc) over its eligible rows, one row per thread: every
// eligible row is ranked against the others (see decide_fast). All threads of the CTA call it.
__device__ __forceinline__ void topk_rank(uint64_t* keys, int seg, int per_seq, int topk, const float* score,
                                          const uint8_t* eligible, int32_t* topk_idx, float* topk_score) {
  const int tid = threadIdx.x, nt = blockDim.x;
  const int base = seg * per_seq;
  uint64_t key = 0;
  float sc = 0.0f;
  if (tid < per_seq) {
    // both loads issued together: the score is read whether or not the row is eligible
    sc = __ldcg(score + base + tid);
    if (eligible == nullptr || eligible[base + tid] != 0) key = rank_key(sc, tid);
  }
  if (tid < per_seq) keys[tid] = key;
  const int n_elig = __syncthreads_count(key != 0);
  const int r = rank_below(keys, per_seq, key, topk);
  if (key != 0 && r < topk) {
    topk_idx[static_cast<size_t>(seg) * topk + r] = tid;
    if (topk_score != nullptr) topk_score[static_cast<size_t>(seg) * topk + r] = sc;
  }
  for (int t = min(n_elig, topk) + tid; t < topk; t += nt) {
    topk_idx[static_cast<size_t>(seg) * topk + t] = -1;
    if (topk_score != nullptr) topk_score[static_cast<size_t>(seg) * topk + t] = -INFINITY;
  }
}

// The keys of a segment of any length in keys[0 .. sort_n).
__device__ __forceinline__ void topk_keys(uint64_t* keys, int seg, int per_seq, int sort_n, const float* score,
                                          const uint8_t* eligible) {
  const int tid = threadIdx.x, nt = blockDim.x;
  const int base = seg * per_seq;
  // the scores and flags of kLoads rows per thread are loaded before any key is stored, so the
  // loads of a thread overlap instead of waiting one after the other
  constexpr int kLoads = 4;
  for (int i0 = tid; i0 < sort_n; i0 += kLoads * nt) {
    float sc[kLoads];
    bool el[kLoads];
#pragma unroll
    for (int u = 0; u < kLoads; ++u) {
      const int i = i0 + u * nt;
      const bool in = i < per_seq;
      sc[u] = in ? __ldcg(score + base + i) : 0.0f;
      el[u] = in && (eligible == nullptr || eligible[base + i] != 0);
    }
#pragma unroll
    for (int u = 0; u < kLoads; ++u) {
      const int i = i0 + u * nt;
      if (i < sort_n) keys[i] = el[u] ? rank_key(sc[u], i) : 0;
    }
  }
  __syncthreads();
}

// Slot `slot` of the lists: the row and score of a key, none for key 0.
__device__ __forceinline__ void topk_put(uint64_t key, size_t slot, int32_t* topk_idx, float* topk_score) {
  topk_idx[slot] = key != 0 ? rank_key_row(key) : -1;
  if (topk_score != nullptr) topk_score[slot] = key != 0 ? order_key_inv(static_cast<uint32_t>(key >> 32)) : -INFINITY;
}

// The last CTA of a segment in a row kernel: ranks where every row has a thread of the bulk-copy kernel's,
// else a list of a few.
__device__ __forceinline__ void segment_topk(uint64_t* keys, int seg, const ScoreParams& P) {
  if (P.per_seq <= kBulkThreads) {
    topk_rank(keys, seg, P.per_seq, P.topk, P.score, P.eligible, P.topk_idx, P.topk_score);
    return;
  }
  __shared__ uint64_t s_few[kFusedTopk];
  topk_keys(keys, seg, P.per_seq, P.sort_n, P.score, P.eligible);
  top_rounds(keys, P.sort_n, P.topk, s_few);
  if (static_cast<int>(threadIdx.x) < P.topk)
    topk_put(s_few[threadIdx.x], static_cast<size_t>(seg) * P.topk + threadIdx.x, P.topk_idx, P.topk_score);
}

// Accumulate U vectors of 8 values; the first index of vector u is i0 + u * istride, istride
// being the kernel's constant batch stride when U > 1.
// Per pair of values: one packed FMA for t, two ex2, one packed add into Z and
// one packed FMA into S; two independent accumulator chains.
template <int U>
__device__ __forceinline__ void acc_batch(RowAcc& a, const uint4 (&w)[U], int i0) {
  float x[U][8];
  float bmax = -INFINITY;
#pragma unroll
  for (int u = 0; u < U; ++u) {
    unpack8(w[u], x[u]);
#pragma unroll
    for (int k = 0; k < 8; k += 2) bmax = fmax3(bmax, x[u][k], x[u][k + 1]);
  }
  // the batch is recorded, not searched: only the row maximum's first index is needed, and
  // row_reduce finds it in the recorded batches of the threads that hold that maximum
  if (bmax > a.m) raise_max(a, bmax, i0, U);
  const uint64_t c2 = f2_pack(kLog2e, kLog2e);
  const uint64_t nm2 = f2_pack(-a.mref, -a.mref);
  uint64_t z[2] = {0, 0}, sacc[2] = {0, 0};
#pragma unroll
  for (int u = 0; u < U; ++u) {
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const uint64_t t2 = f2_fma(f2_pack(x[u][2 * k], x[u][2 * k + 1]), c2, nm2);
      float t0, t1;
      f2_unpack(t2, t0, t1);
      const uint64_t e2 = f2_pack(ex2_approx(t0), ex2_approx(t1));
      z[k & 1] = f2_add(z[k & 1], e2);
      sacc[k & 1] = f2_fma(t2, e2, sacc[k & 1]);
    }
  }
  float z0, z1, s0, s1;
  f2_unpack(f2_add(z[0], z[1]), z0, z1);
  f2_unpack(f2_add(sacc[0], sacc[1]), s0, s1);
  kahan_add(a.z, a.zc, z0 + z1);
  kahan_add(a.s, a.sc, s0 + s1);
}


// ---------------------------------------------------------------------------
// row kernel: bulk copies of a row, or of a row's slice in each CTA of a cluster
// ---------------------------------------------------------------------------
// L2 policy of the copies: evicted first where the logits are not read again, which leaves the rest of a
// step there (states, weights, the next kernels' code). That is a decision step's, whose launches went from
// 98.9 to 87.2 us in Dream's shape (311 MB of logits) and from 39.5 to 33.8 with 28 / 4 heads, 243 rows (74
// MB), and plain scoring of more than L2 holds. Other plain scoring leaves the logits there: evicted first,
// a second call on 1024 rows of 32000 logits took 16.9 instead of 13.9 us, of 50000 22.3 instead of 20.2, and
// calls on three 21 MB sets in turn 10.1 instead of 8.9. The pass itself takes the same time either way.
__device__ __forceinline__ uint64_t stream_policy(bool evict_first) {
  uint64_t p;
  if (evict_first)
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
  else
    asm volatile("createpolicy.fractional.L2::evict_normal.b64 %0, 1.0;" : "=l"(p));
  return p;
}
__device__ __forceinline__ void bulk_load(void* smem_dst, const void* src, uint32_t bytes, uint64_t* bar,
                                          uint64_t policy) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint"
      " [%0], [%1], %2, [%3], %4;" ::"r"(smem_u32(smem_dst)),
      "l"(src), "r"(bytes), "r"(smem_u32(bar)), "l"(policy)
      : "memory");
}

// Writes r to *dst of the cluster's CTA `rank` (dst: this CTA's copy of the same variable).
__device__ __forceinline__ void cluster_store_row_sum(RowSum* dst, uint32_t rank, const RowSum& r) {
  const uint32_t d = cluster_map(smem_u32(dst), rank);
  asm volatile(
      "st.shared::cluster.v2.f32 [%0], {%1, %2};\n\t"
      "st.shared::cluster.v2.f32 [%0 + 8], {%3, %4};\n\t"
      "st.shared::cluster.v2.f32 [%0 + 16], {%5, %6};" ::"r"(d),
      "f"(r.M), "f"(__int_as_float(r.yhat)), "f"(r.zh), "f"(r.zl), "f"(r.sh), "f"(r.sl)
      : "memory");
}

template <int C>
__global__ void __launch_bounds__(kBulkThreads, 4) score_bulk_kernel(const ScoreParams P, int* status) {
  extern __shared__ __align__(128) uint8_t dsmem[];   // ring, reused for top-k keys
  __shared__ uint64_t bar_full[kRingStages], bar_empty[kRingStages];
  __shared__ float red_m[kConsumerWarps + 1];
  __shared__ int red_i[kConsumerWarps + 1];
  __shared__ float2 red_z[kConsumerWarps + 1], red_s[kConsumerWarps + 1];
  __shared__ int s_last, s_abort;
  __shared__ RowSum s_part[C];   // the cluster's slice sums, in its first CTA
  __shared__ RowSide s_side;
  if (C > 1) cluster_arrive();   // completed before the slice sums are sent: every CTA has started
  // programmatic dependent launch: wait for the stream's previous kernel, let the next one be
  // scheduled
  griddep_wait();
  griddep_launch_dependents();

  const int n = blockIdx.x / C;
  const int rank = C > 1 ? static_cast<int>(cluster_ctarank()) : 0;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int V = P.V;
  const size_t row_off = static_cast<size_t>(n) * V;
  const uint16_t* row = P.logits + row_off;
  // the row's aligned 16-byte vectors go through the ring, the few elements before and after
  // them are read directly
  const int head = min(static_cast<int>((8 - (row_off & 7)) & 7), V);
  const int row_vec = (V - head) / 8;
  const int slice = C > 1 ? (row_vec + C - 1) / C : row_vec;
  const int first = head + min(rank * slice, row_vec) * 8;   // first element of this CTA's slice
  const int elems_all = min(slice, row_vec - min(rank * slice, row_vec)) * 8;
  const int nchunks = (elems_all + kChunkElems - 1) / kChunkElems;
  const uint16_t* src_row = row + first;
  uint8_t* ring = dsmem;
  const uint64_t policy = stream_policy(P.evict_first);

  if (warp == kConsumerWarps && lane == 0) {
    // the producer initialises the ring and issues its first chunks at once, so their latency
    // overlaps the block barrier
    for (int s = 0; s < kRingStages; ++s) {
      mbar_init(&bar_full[s], 1);
      mbar_init(&bar_empty[s], kConsumerWarps);
    }
    s_abort = 0;
    fence_mbar_init();
    for (int c = 0; c < kRingStages && c < nchunks; ++c) {
      const int elems = min(kChunkElems, elems_all - c * kChunkElems);
      mbar_arrive_expect_tx(&bar_full[c], static_cast<uint32_t>(elems * 2));
      bulk_load(ring + c * kChunkBytes, src_row + static_cast<size_t>(c) * kChunkElems,
                static_cast<uint32_t>(elems * 2), &bar_full[c], policy);
    }
  }
  __syncthreads();

  RowAcc a{-INFINITY, 0x7fffffff, 0, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
  if (warp == kConsumerWarps) {
    // producer: one lane streams the row chunk by chunk
    if (lane == 0) {
      // the row's side data, on its way while the row streams (its logit once the token is here)
      RowSide side{true, 0.0f, 0.0f, 0.0f};
      int y = 0;
      if (rank == 0) {
        const int32_t* tok = P.decide ? P.dec.tok : P.cur_tok;
        side.greedy = tok == nullptr;
        if (tok != nullptr) y = tok[n];
        if (!P.decide && P.d_in != nullptr) side.din = P.d_in[n];
        if (!P.decide && P.d_out != nullptr) side.dout = P.d_out[n];
      }
      if (nchunks <= kRingStages) side_logit(side, y, row, V);
      for (int c = kRingStages; c < nchunks; ++c) {
        const int st = c % kRingStages;
        if (!mbar_wait(&bar_empty[st], ((c / kRingStages) - 1) & 1, &s_abort)) {
          report_status(status, kStatusTimeout, 200);
          s_abort = 1;
          break;
        }
        const int elems = min(kChunkElems, elems_all - c * kChunkElems);
        mbar_arrive_expect_tx(&bar_full[st], static_cast<uint32_t>(elems * 2));
        bulk_load(ring + st * kChunkBytes, src_row + static_cast<size_t>(c) * kChunkElems,
                  static_cast<uint32_t>(elems * 2), &bar_full[st], policy);
        if (c == kRingStages) side_logit(side, y, row, V);
      }
      s_side = side;
      // every copy issued has been consumed once the consumers pass their last
      // full-barrier wait; nothing is left in flight at the final barrier
    } else if (rank == 0 && lane <= 16) {
      // the elements outside the aligned vectors: lanes 1 .. 8 before them, 9 .. 16 after them
      const int i = lane <= 8 ? lane - 1 : head + row_vec * 8 + lane - 9;
      if (lane <= 8 ? i < head : i < V) acc_scalar(a, bf16_to_f32(row[i]), i);
    }
  } else {
    for (int c = 0; c < nchunks; ++c) {
      const int st = c % kRingStages;
      const bool ok = mbar_wait(&bar_full[st], (c / kRingStages) & 1, &s_abort);
      if (!__all_sync(0xffffffffu, ok)) {
        if (lane == 0) {
          report_status(status, kStatusTimeout, 201);
          s_abort = 1;
        }
        break;
      }
      const int elems = min(kChunkElems, elems_all - c * kChunkElems);
      const uint4* src = reinterpret_cast<const uint4*>(ring + st * kChunkBytes);
      const int nv = elems / 8;
      constexpr int kStride = kConsumerWarps * 32;
      if (tid + (kVecPerThread - 1) * kStride < nv) {
        uint4 w[kVecPerThread];
#pragma unroll
        for (int u = 0; u < kVecPerThread; ++u) w[u] = src[tid + u * kStride];
        acc_batch<kVecPerThread>(a, w, first + c * kChunkElems + tid * 8);
      } else {
        for (int v = tid; v < nv; v += kStride) {
          uint4 w[1] = {src[v]};
          acc_batch<1>(a, w, first + c * kChunkElems + v * 8);
        }
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(&bar_empty[st]);
    }
  }
  // if the producer gave up, wait (bounded) for the copies it already issued
  if (warp == kConsumerWarps && lane == 0 && s_abort) {
    for (int c = max(0, nchunks - kRingStages); c < nchunks; ++c)
      mbar_wait(&bar_full[c % kRingStages], (c / kRingStages) & 1, nullptr, 1000000ull);
  }
  __syncwarp();

  const Ring held{ring, first, nchunks - kRingStages};
  RowSum r = row_reduce<kConsumerWarps + 1, kConsumerWarps * 32 * 8>(a, row, held, red_m, red_i, red_z, red_s);
  if (C > 1) {
    // every CTA sends its slice's sums to the cluster's first, which adds them
    __syncwarp();
    cluster_wait();
    if (tid == 0) cluster_store_row_sum(&s_part[rank], 0, r);
    __syncwarp();
    cluster_arrive();
    if (rank != 0) return;
    cluster_wait();
    if (warp == 0) r = row_combine<C>(s_part, lane);
  }
  if (tid == 0)
    s_last = row_write(row_finish(r), s_side, n, P.per_seq, P.topk, P.maxprob, P.entropy, P.argmax, P.score,
                       P.decide == kDecideApart ? nullptr : P.counters, P.decide ? P.dec.ws_u : nullptr,
                       P.decide ? P.dec.ws_lnz : nullptr);
  __syncthreads();
  if (s_last) {
    if (P.decide)
      decide_fast<false>(reinterpret_cast<uint64_t*>(ring), n / P.per_seq, P.per_seq, P);
    else
      segment_topk(reinterpret_cast<uint64_t*>(ring), n / P.per_seq, P);
  }
}

// Rows that do not start on 16-byte boundaries (V % 8 != 0), a few of them per SM: a CTA's 16 warps load
// the row's aligned vectors into registers, and the elements before and after them.
__global__ void __launch_bounds__(kRegThreads, 2) score_reg_kernel(const ScoreParams P) {
  extern __shared__ __align__(16) uint64_t reg_keys[];
  constexpr int kWarps = kRegThreads / 32;
  __shared__ float red_m[kWarps];
  __shared__ int red_i[kWarps];
  __shared__ float2 red_z[kWarps], red_s[kWarps];
  __shared__ int s_last;
  griddep_wait();
  griddep_launch_dependents();

  const int n = blockIdx.x, tid = threadIdx.x, V = P.V;
  const size_t row_off = static_cast<size_t>(n) * V;
  const uint16_t* row = P.logits + row_off;
  // the row's side data, on its way while the row streams; the token's logit once the row is read
  RowSide side{true, 0.0f, 0.0f, 0.0f};
  int y = 0;
  if (tid == 0) {
    const int32_t* tok = P.decide ? P.dec.tok : P.cur_tok;
    side.greedy = tok == nullptr;
    if (tok != nullptr) y = tok[n];
    if (!P.decide && P.d_in != nullptr) side.din = P.d_in[n];
    if (!P.decide && P.d_out != nullptr) side.dout = P.d_out[n];
  }
  RowAcc a{-INFINITY, 0x7fffffff, 0, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
  const int head = min(static_cast<int>((8 - (row_off & 7)) & 7), V);
  const int nvec = (V - head) / 8, tail0 = head + nvec * 8;
  if (tid < head) acc_scalar(a, bf16_to_f32(row[tid]), tid);
  const uint4* vrow = reinterpret_cast<const uint4*>(row + head);
  int v = tid;
  for (; v + (kRegUnroll - 1) * kRegThreads < nvec; v += kRegUnroll * kRegThreads) {
    uint4 w[kRegUnroll];
#pragma unroll
    for (int u = 0; u < kRegUnroll; ++u) w[u] = ld_stream(vrow + v + u * kRegThreads);
    acc_batch<kRegUnroll>(a, w, head + v * 8);
  }
  for (; v < nvec; v += kRegThreads) {
    uint4 w[1] = {ld_stream(vrow + v)};
    acc_batch<1>(a, w, head + v * 8);
  }
  if (tail0 + tid < V) acc_scalar(a, bf16_to_f32(row[tail0 + tid]), tail0 + tid);
  if (tid == 0) side_logit(side, y, row, V);

  const Ring none{nullptr, 0, 0x7fffffff};
  const RowSum r = row_reduce<kWarps, kRegThreads * 8>(a, row, none, red_m, red_i, red_z, red_s);
  if (tid == 0)
    s_last = row_write(row_finish(r), side, n, P.per_seq, P.topk, P.maxprob, P.entropy, P.argmax, P.score,
                       P.decide == kDecideApart ? nullptr : P.counters, P.decide ? P.dec.ws_u : nullptr,
                       P.decide ? P.dec.ws_lnz : nullptr);
  __syncthreads();
  if (s_last) {
    if (P.decide)
      decide_fast<false>(reg_keys, n / P.per_seq, P.per_seq, P);
    else
      segment_topk(reg_keys, n / P.per_seq, P);
  }
}

// One step's decisions as their own launch (one CTA per segment) behind the row kernel, for segments
// of more rows than that kernel's CTAs have threads: up to 1024 rows then have a thread each, where
// the last CTA of a segment made five passes over its rows. Segments of up to kBulkThreads rows
// stay in the row kernel, where the last CTA starts on them at once.
// 1 x 1024 rows of 152064 logits: 70.6 -> 62.0 us (54.0 us for the rows alone), and 92 -> 68 us in a
// decoding step, whose other launches leave the row state in L2 only.
__global__ void __launch_bounds__(kMaxThreads) decide_kernel(const ScoreParams P) {
  extern __shared__ __align__(16) uint64_t dec_keys[];
  griddep_wait();
  griddep_launch_dependents();
  segment_decide(dec_keys, blockIdx.x, P.per_seq, P.sort_n, P);
}

// The top-k of such segments, likewise, for lists of more than kFusedTopk. Shorter ones stay with the row
// kernel's last CTA: rounds take it about as long as the second launch takes this kernel (600 rows of 1001
// logits, k = 1 / 8: 6.3 / 8.3 us against 6.7 / 6.7), and a call of little work is bound by the host, where the
// launch costs 2 us. How, by the rows and the list, with the us that the launch adds behind rows of 1001
// logits:
//   rows           list       merged lists   ranks             warp sorts, 288 / 512 / 1024 threads   sort, 512 / 1024
//   289            <= 32      2.6            3.9               6.1 / 6.9                              9.4 / 10.2
//   289, 400, 512  33 .. 200                 3.9, 5.4, 6.3                                            9.4, 9.6, 9.5 / 10.2, 9.8, 10.5
//   640, 768, 1024 33 .. 200                 9.3, 13.0, 21.7                                          17.3, 17.5, 17.8 / 14.1, 14.3, 14.4
//   1024           <= 32      3.6            21.7              6.1 / 8.4 / 16.1
//   2048           <= 32                                       8.6 / 8.1 / 16.2
//   4096           <= 32                                       14.2 / 12.0 / 16.5
// In the row kernel's last CTA of 288 threads, lists of more than 32 rows were sorted: 1 x 512 rows of 20001
// logits, k = 64: 20.7 us; a row kernel of 512 threads ranked them: 16.4; now 13.3 (1024 rows: 39.3, 35.2, 25.3).
constexpr int kRankRows = 768;        // segments up to this size are ranked, for lists of more than kRoundsMax
constexpr int kTopkWarpThreads = 512; // threads for a short list of more rows than a CTA can have threads
int topk_threads(int per, int topk) {
  const bool list = topk <= kRoundsMax;
  if (per > kMaxThreads) return list ? kTopkWarpThreads : kMaxThreads;
  return list || per <= kRankRows ? (per + 31) / 32 * 32 : kMaxThreads;
}
__global__ void __launch_bounds__(kMaxThreads) topk_kernel(const ScoreParams P) {
  extern __shared__ __align__(16) uint64_t topk_smem[];
  __shared__ uint64_t s_sel[kRoundsMax];
  griddep_wait();
  griddep_launch_dependents();
  const int tid = threadIdx.x, nt = blockDim.x, seg = blockIdx.x;
  const size_t list = static_cast<size_t>(seg) * P.topk;
  if (P.per_seq <= nt && P.topk <= kRoundsMax) {
    uint64_t key = 0;
    if (tid < P.per_seq) {
      const int n = seg * P.per_seq + tid;
      const float sc = P.score[n];
      if (P.eligible == nullptr || P.eligible[n] != 0) key = rank_key(sc, tid);
    }
    const uint64_t held = top_merged(warp_sort_desc(key, tid & 31), topk_smem);
    if (tid < P.topk) topk_put(held, list + tid, P.topk_idx, P.topk_score);
  } else if (P.per_seq <= nt && P.per_seq <= kRankRows) {
    topk_rank(topk_smem, seg, P.per_seq, P.topk, P.score, P.eligible, P.topk_idx, P.topk_score);
  } else {
    const uint64_t* best = topk_smem;
    topk_keys(topk_smem, seg, P.per_seq, P.sort_n, P.score, P.eligible);
    if (P.topk <= kRoundsMax) {
      top_warps(topk_smem, P.sort_n, P.topk, s_sel);
      best = s_sel;
    } else {
      bitonic_sort_desc(topk_smem, P.sort_n);
    }
    for (int t = tid; t < P.topk; t += nt) topk_put(best[t], list + t, P.topk_idx, P.topk_score);
  }
}

// Section 5.3 selection as its own launch (one CTA per segment), after the
// update phase and the d_in / d_out pass.
constexpr int kSelectThreads = 512;
static_assert(kBulkThreads <= 32 * kMaxWarps && kSelectThreads <= 32 * kMaxWarps,
              "top_rounds keeps a list per warp for at most kMaxWarps warps");
__global__ void __launch_bounds__(kSelectThreads) seed_select_kernel(const DecideArgs d, const float* d_in,
                                                                    const float* d_out, float* score, int per_seq,
                                                                    int sort_n) {
  extern __shared__ __align__(16) uint64_t sel_keys[];
  // programmatic dependent launch: wait for the stream's previous kernel, let the next one be
  // scheduled
  griddep_wait();
  griddep_launch_dependents();
  const int tid = threadIdx.x;
  if (per_seq <= static_cast<int>(blockDim.x)) {
    // one row per thread: the state in registers, selection by rank
    const int n = blockIdx.x * per_seq + tid;
    const bool in = tid < per_seq;
    int tok = 0;
    uint32_t fl = 0, rc = 0;
    float u = 0.0f, din = 0.0f, dout = 0.0f;
    if (in) {
      tok = d.tok[n];
      fl = d.flags[n];
      rc = d.remask_cnt[n];
      u = d.ws_u[n];
      din = d_in != nullptr ? d_in[n] : 0.0f;
      dout = d_out != nullptr ? d_out[n] : 0.0f;
    }
    select_fast<false>(sel_keys, blockIdx.x, per_seq, d, in, tok, fl, rc, u, din, dout, score);
    if (in) d.flags[n] = static_cast<uint8_t>(fl);
    return;
  }
  segment_select(sel_keys, blockIdx.x, per_seq, sort_n, d, d_in, d_out, score);
}

}  // namespace

namespace {

template <int C>
int launch_rows(const ScoreParams& P, int N, size_t smem, int* status, cudaStream_t stream) {
  // the ring's shared-memory limit is a function attribute of the current context
  static ContextCache<int> setup;
  int unused = 0;
  const int rc = setup.get(&unused, [](int&) {
    return cudaFuncSetAttribute(score_bulk_kernel<C>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                static_cast<int>(kRingStages * kChunkBytes)) == cudaSuccess ? 0 : -3;
  });
  if (rc != 0) return rc;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = C;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(static_cast<unsigned>(N) * C);
  cfg.blockDim = dim3(kBulkThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cfg.attrs = attr;
  cfg.numAttrs = C > 1 ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, score_bulk_kernel<C>, P, status) == cudaSuccess ? 0 : -3;
}

// CTAs a row is split over. A row alone on an SM is bound by its own CTA (12 us at V = 126464), so
// few rows are split until the launch holds two CTAs per SM. Beyond that the SMs' issue rate is
// shared anyway and every further CTA only adds its start and reduction. us at 1 / 2 / 4 / 8 CTAs a
// row, V = 126464: 32 rows 12.5 / 9.2 / 7.4 / 6.8, 64 rows 12.7 / 9.5 / 8.5 / 8.9, 128 rows 13.6 / 12.0
// / 12.4 / 15.9, 152 rows 14.7 / 13.4 / 17.3 / 20.2, 200 rows 17.8 / 18.4 / 22.1 / 24.2. V = 32000:
// 32 rows 6.4 / 6.3 / 5.9 / 5.5, 128 rows 7.0 / 7.2 / 7.7 / 11.5: halves of a short row do not pay. Where they
// begin to, 1 / 2 CTAs a row: 100 rows of 60000 7.7 / 7.8, of 65536 7.7 / 7.7, of 80000 9.1 / 8.5; 152 rows 8.1 /
// 8.3, 8.2 / 8.2, 9.6 / 9.2. Two CTAs a row that do not fit two to an SM: 154 rows of 80000 10.9 / 12.0, of 126464
// 14.6 / 15.3.
int row_split(int N, int V, int n_sm) {
  int c = kMaxSplit;
  while (c > 1 && (static_cast<long long>(N) * c > 2LL * n_sm || V < c * kMinSlice || (c == 2 && V < 65536))) c >>= 1;
  return c;
}

// Whether unaligned rows go through the register-load kernel: with one or two unsplit rows per SM its 16
// warps are ahead of the ring's 8, except where much of a short row is left over whole batches of its CTA
// (16384 elements; the rest goes a vector at a time). us through the ring / registers, by rows and V:
//   rows   18435      20001      26001      30001      36355      45001      48001      53001      65001
//   100    4.2 / 3.8  4.3 / 4.0  4.8 / 4.7  5.1 / 5.1  5.8 / 5.3  6.6 / 6.7  6.9 / 7.5  7.3 / 6.7  7.9 / 7.9
//   153    4.7 / 5.0  5.0 / 5.2  5.8 / 6.5  6.6 / 7.8  7.2 / 6.6  7.9 / 7.9  8.4 / 8.4  8.6 / 7.8  9.5 / 9.1
//   250    6.0 / 5.9  6.3 / 6.0  7.0 / 7.3  7.5 / 8.4  8.0 / 7.1  8.7 / 8.4  9.2 / 9.1  9.5 / 8.6  10.3 / 9.9
//   rows   78001        85001        90125        95001        99001        113001       130001       152065
//   153    10.7 / 10.6  11.4 / 10.3  11.7 / 11.0  12.1 / 12.2  12.4 / 11.0  13.5 / 12.9  15.0 / 13.6  16.8 / 15.6
//   250    11.5 / 11.6  12.2 / 11.2  12.6 / 12.1  13.0 / 13.4  13.2 / 12.2  14.4 / 14.0  15.9 / 15.0  17.8 / 16.9
// and with more rows 320 of 20001 8.2 / 8.9, of 50257 12.8 / 12.9, of 152065 27.8 / 27.0; 153 of 8001 4.0 / 4.1.
bool loads_to_registers(int N, int V, int split, int n_sm) {
  constexpr int kBatch = kRegThreads * kRegUnroll * 8;
  const int left = V % kBatch;
  return V % 8 != 0 && split == 1 && N <= 2 * n_sm &&
         (V >= 6 * kBatch || (V >= 2 * kBatch && left <= 3 * kBatch / 4) || (V >= 9 * kBatch / 8 && left <= kBatch / 4));
}

int launch_score_impl(const ScoreArgs& a, const DecideArgs* d, int* status, cudaStream_t stream) {
  struct Device {
    int n_sm, l2_bytes;
  };
  static ContextCache<Device> devices;
  Device gpu{};
  const int rc = devices.get(&gpu, [](Device& v) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return -3;
    return cudaDeviceGetAttribute(&v.n_sm, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess &&
                   cudaDeviceGetAttribute(&v.l2_bytes, cudaDevAttrL2CacheSize, dev) == cudaSuccess ? 0 : -3;
  });
  if (rc != 0) return rc;
  const int n_sm = gpu.n_sm;
  const int per = a.N / a.n_seq;
  int sort_n = 1;
  while (sort_n < per) sort_n <<= 1;
  ScoreParams P{static_cast<const uint16_t*>(a.logits), a.V, per, a.cur_tok, a.d_in, a.d_out, a.eligible,
                a.topk, sort_n, a.maxprob, a.entropy, a.argmax, a.score, a.topk_idx, a.topk_score, a.counters,
                d == nullptr ? 0 : per > kBulkThreads ? kDecideApart : kDecideFused, d != nullptr ? *d : DecideArgs{},
                d != nullptr || 2LL * a.N * a.V > gpu.l2_bytes};
  // top-k keys (at most 4096 x 8 bytes) reuse the ring; so does the decision step, which keeps a
  // float score per row behind them (4096 x 12 bytes, exactly the ring)
  static_assert((sizeof(uint64_t) + sizeof(float)) * kMaxPerSeq <= kRingStages * kChunkBytes, "keys fit the ring");
  const size_t smem = static_cast<size_t>(kRingStages) * kChunkBytes;
  const bool long_topk = d == nullptr && a.topk > kFusedTopk && per > kBulkThreads;
  ScoreParams rows = P;
  if (long_topk) rows.topk = 0;
  int rl = 0;
  const int split = row_split(a.N, a.V, n_sm);
  if (loads_to_registers(a.N, a.V, split, n_sm)) {
    cudaLaunchAttribute attr[1];
    const cudaLaunchConfig_t cfg = pdl_config(dim3(static_cast<unsigned>(a.N)), dim3(kRegThreads),
                                              sizeof(uint64_t) * std::max(sort_n, kRegThreads), stream, attr);
    rl = cudaLaunchKernelEx(&cfg, score_reg_kernel, rows) == cudaSuccess ? 0 : -3;
  } else {
    switch (split) {
      case 8: rl = launch_rows<8>(rows, a.N, smem, status, stream); break;
      case 4: rl = launch_rows<4>(rows, a.N, smem, status, stream); break;
      case 2: rl = launch_rows<2>(rows, a.N, smem, status, stream); break;
      default: rl = launch_rows<1>(rows, a.N, smem, status, stream);
    }
  }
  if (rl != 0 || (!long_topk && P.decide != kDecideApart)) return rl;
  const int threads = long_topk ? topk_threads(per, a.topk) : std::min((per + 31) / 32 * 32, kMaxThreads);
  const size_t keys = (sizeof(uint64_t) + (long_topk ? 0 : sizeof(float))) * static_cast<size_t>(std::max(sort_n, threads));
  static ContextCache<int> setup;
  int unused = 0;
  const int rc2 = setup.get(&unused, [](int&) {
    return cudaFuncSetAttribute(decide_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                static_cast<int>((sizeof(uint64_t) + sizeof(float)) * kMaxPerSeq)) == cudaSuccess
               ? 0 : -3;
  });
  if (rc2 != 0) return rc2;
  cudaLaunchAttribute attr[1];
  const cudaLaunchConfig_t cfg = pdl_config(dim3(static_cast<unsigned>(a.n_seq)), dim3(threads), keys, stream, attr);
  return cudaLaunchKernelEx(&cfg, long_topk ? topk_kernel : decide_kernel, P) == cudaSuccess ? 0 : -3;
}

}  // namespace

int launch_score(const ScoreArgs& a, int* status, cudaStream_t stream) {
  return launch_score_impl(a, nullptr, status, stream);
}

int launch_score_decide(const ScoreArgs& a, const DecideArgs& d, int* status, cudaStream_t stream) {
  return launch_score_impl(a, &d, status, stream);
}

int launch_seed_select(int N, int n_seq, const DecideArgs& d, const float* d_in, const float* d_out, float* score,
                       cudaStream_t stream) {
  const int per = N / n_seq;
  int sort_n = 1;
  while (sort_n < per) sort_n <<= 1;
  // at least one key per thread: the one-row-per-thread selection publishes up to 32 keys per warp
  const size_t smem = (sizeof(uint64_t) + sizeof(float)) * static_cast<size_t>(std::max(sort_n, kSelectThreads));
  // the longest segment's keys and scores (48 KB) need the opt-in above the default limit
  static ContextCache<int> setup;
  int unused = 0;
  const int rc = setup.get(&unused, [](int&) {
    return cudaFuncSetAttribute(seed_select_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                static_cast<int>((sizeof(uint64_t) + sizeof(float)) * kMaxPerSeq)) == cudaSuccess
               ? 0 : -3;
  });
  if (rc != 0) return rc;
  cudaLaunchAttribute attr[1];
  const cudaLaunchConfig_t cfg = pdl_config(dim3(n_seq), dim3(kSelectThreads), smem, stream, attr);
  if (cudaLaunchKernelEx(&cfg, seed_select_kernel, d, d_in, d_out, score, per, sort_n) != cudaSuccess) return -3;
  return cudaGetLastError() == cudaSuccess ? 0 : -3;
}

// ---------------------------------------------------------------------------
// Allocation-free variant: the same kernels, with the per-segment counters in
// a fixed device array of this library instead of a caller workspace.
// ---------------------------------------------------------------------------
namespace {

// Counters for at most kNoAllocMaxSegments segments (16 KB). Every device that
// loads the library holds one copy until the process exits.
static __device__ __align__(256) uint32_t g_noalloc_counters[kNoAllocMaxSegments];

// Device address of the counter array in the current device's context. In host
// code the array's name is only a host-side stand-in, so the address is looked up
// (cudaGetSymbolAddress, with the device current) the first time a context calls,
// and again in a context created anew after cudaDeviceReset.
uint32_t* noalloc_counters() {
  static ContextCache<uint32_t*> cache;
  uint32_t* p = nullptr;
  const int rc = cache.get(&p, [](uint32_t*& v) {
    void* a = nullptr;
    if (cudaGetSymbolAddress(&a, g_noalloc_counters) != cudaSuccess || a == nullptr) return -3;
    v = static_cast<uint32_t*>(a);
    return 0;
  });
  return rc == 0 ? p : nullptr;
}

}  // namespace

int launch_score_noalloc(ScoreArgs a, int* status, cudaStream_t stream) {
  if (a.n_seq > kNoAllocMaxSegments) return -1;
  uint32_t* counters = noalloc_counters();
  if (counters == nullptr) return -3;
  // the array keeps whatever the previous call left: the counters this call
  // uses must start at zero
  if (a.topk > 0 &&
      cudaMemsetAsync(counters, 0, sizeof(uint32_t) * static_cast<size_t>(a.n_seq), stream) != cudaSuccess)
    return -3;
  a.counters = counters;
  return launch_score(a, status, stream);
}

}  // namespace cover
