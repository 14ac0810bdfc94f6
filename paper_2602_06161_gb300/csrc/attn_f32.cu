// attn_f32.cu - two-view override attention in fp32 on CUDA cores.
//
// Section 5.1: every query attends once over the overridden memory K', V'
// (scale 1/sqrt(d)); a seed query i sees its diagonal entry restored to the
// masked-input pair (k_i, v_i). The kernel applies Appendix B's diagonal
// correction in exclusion form: the cached diagonal term (k'_i, v'_i) is left
// out of the online softmax, and the masked self term is merged into the
// running (max, sum, output) at the end. In exact arithmetic this equals the
// closed form o_i = (o_ovr_i - alpha_i v'_i + alpha_i e^delta_i v_i) / r_i,
// without its division by r_i (which tends to 0 as alpha_i -> 1 and
// delta_i -> -inf).
//
// A CTA of four warps takes BM = 16 TM query rows of one head against key tiles of 64. Thread
// (ty, tx) of the 16 x 8 arrangement holds rows 16 w + 4 i + ty % 4 (i < TM, w the warp) and, of a
// score tile, keys tx + 8 j, of the output, columns 4 tx + 32 c .. + 3: a warp owns its 4 TM rows
// through both products, so the probabilities pass through shared memory within the warp and the
// row statistics are eight-lane shuffles.
//
// Bound: the register ports of the fp32 FMAs. 4 B Hq Lq L D flops at the pipe's 128 FMA/clk/SM
// (76 TFLOP/s at 1.95 GHz) are the floor (tensor cores would round the operands), but an FMA whose
// three operands all come from the register file takes about 1.4 issue slots instead of 1, packed
// f32x2 (2.8 for two, measured) or not. The packed form leaves issue slots for the rest of the
// loop: 118 against 143 us with scalar FMAs on 32 heads x 512 rows x 512 keys, D = 128 (36 TFLOP/s;
// one warp per row with a shuffle reduction per key took 1140 us). Two other layouts measured the
// same there: eight warps with half the register tile (125 us), and lanes whose shared-memory reads
// do not merge (124 us).
#include <math.h>

#include "cluster.cuh"
#include "context.cuh"
#include "kernels.cuh"
#include "ptx.cuh"
#include "route.cuh"

namespace cover {
namespace {

constexpr int kThreads = 128;
constexpr int kBN = 64;    // keys per tile

template <int D, int TM>
struct F32Tile {
  static constexpr int kBM = 16 * TM;
  static constexpr int kQ = kBM * D, kKV = kBN * D, kP = kBM * kBN;   // floats
  static constexpr size_t kBytes = sizeof(float) * (kQ + 2 * kKV + kP) + sizeof(int) * kBM;
};

__device__ __forceinline__ void cp_async16(uint32_t dst, const float* src, bool in) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(in ? 16 : 0) : "memory");
}
__device__ __forceinline__ void cp_async4(uint32_t dst, const float* src, bool in) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src), "r"(in ? 4 : 0) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

__device__ __forceinline__ ulonglong2 lds2(const float* p) { return *reinterpret_cast<const ulonglong2*>(p); }

// Copies rows [0, ROWS) of D floats at src to shared memory; rows from `valid` on become zeros.
// Swizzled, row r's 16-byte chunk c lands in chunk c ^ (r & 7). Without 16-byte alignment of src
// (vec false) the same chunks go as four 4-byte copies.
template <int D, int ROWS, bool kSwizzle>
__device__ __forceinline__ void load_rows(float* dst, const float* __restrict__ src, int valid, bool vec) {
  constexpr int kChunks = ROWS * D / 4;
  const uint32_t base = smem_u32(dst);
  for (int t = threadIdx.x; t < kChunks; t += kThreads) {
    const int r = t / (D / 4), c = t % (D / 4);
    const bool in = r < valid;
    const float* g = src + (in ? static_cast<size_t>(r) * D + 4 * c : 0);
    const uint32_t d = base + static_cast<uint32_t>(r * D + 4 * (kSwizzle ? c ^ (r & 7) : c)) * 4u;
    if (vec) {
      cp_async16(d, g, in);
    } else {
#pragma unroll
      for (int e = 0; e < 4; ++e) cp_async4(d + 4 * e, g + (in ? e : 0), in);
    }
  }
}

__device__ __forceinline__ float4 ld_cluster4(uint32_t addr) {
  float4 v;
  asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
               : "r"(addr)
               : "memory");
  return v;
}
__device__ __forceinline__ float2 ld_cluster2(uint32_t addr) {
  float2 v;
  asm volatile("ld.shared::cluster.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(addr) : "memory");
  return v;
}

// A whole warp writes row `row` of head `head` again, its keys one by one and the excluded one left out.
// The tiled loop gives that key p = 0, which drops its term only if its cached value row is finite; a
// seed row whose result is not comes here, after the rest. (32 heads x 512 x 512, D = 128: 118.4 against
// 117.0 us without the check, the tiled loop being scheduled otherwise; leaving the term out in that loop
// took 124.8, going through the keys again before the epilogue 122.5.)
template <int D>
__device__ __noinline__ void redo_seed_row(const float* __restrict__ q, const float* __restrict__ kc,
                                           const float* __restrict__ vc, const float* __restrict__ km,
                                           const float* __restrict__ vm, int n_seeds, int Hq, int Hkv, int Lq, int L,
                                           int q0, unsigned head, int row, int slot, float* __restrict__ out,
                                           float* __restrict__ lse) {
  constexpr int E = D / 32;
  const int lane = threadIdx.x & 31;
  const size_t kv_head = static_cast<size_t>(head / static_cast<unsigned>(Hq)) * Hkv +
                         static_cast<int>(head % static_cast<unsigned>(Hq)) / (Hq / Hkv);
  const size_t at = (static_cast<size_t>(head) * Lq + row) * D + lane;
  const float scale = 1.0f / sqrtf(static_cast<float>(D));
  float qr[E], acc[E];
#pragma unroll
  for (int e = 0; e < E; ++e) {
    qr[e] = q[at + 32 * e];
    acc[e] = 0.0f;
  }
  float m = -INFINITY, l = 0.0f;
#pragma unroll 1
  for (int j = 0; j <= L; ++j) {   // j == L: the masked-input pair
    if (j == q0 + row) continue;
    const bool self = j == L;
    const size_t src = (self ? kv_head * n_seeds + slot : kv_head * L + j) * D + lane;
    const float* const kr = (self ? km : kc) + src;
    const float* const vr = (self ? vm : vc) + src;
    float dot = 0.0f;
#pragma unroll
    for (int e = 0; e < E; ++e) dot = fmaf(qr[e], kr[32 * e], dot);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) dot += __shfl_xor_sync(0xffffffffu, dot, o);
    const float s = dot * scale;
    const float m_new = fmaxf(m, s);
    const float a = m == -INFINITY ? 0.0f : expf(m - m_new);
    const float p = expf(s - m_new);
    l = l * a + p;
#pragma unroll
    for (int e = 0; e < E; ++e) acc[e] = acc[e] * a + p * vr[32 * e];
    m = m_new;
  }
  const float inv = 1.0f / l;
#pragma unroll
  for (int e = 0; e < E; ++e) out[at + 32 * e] = acc[e] * inv;
  if (lse != nullptr && lane == 0) lse[static_cast<size_t>(head) * Lq + row] = m + logf(l);
}

// C > 1: the keys of a row tile are split over the C CTAs of a cluster. Each leaves its (m, l, O) in
// its own shared memory, and CTA k combines rows k, k + C, ... from all of them.
template <int D, int TM, int C>
__global__ void __launch_bounds__(kThreads, 2)
    attn_f32_kernel(const float* __restrict__ q, const float* __restrict__ kc, const float* __restrict__ vc,
                    const float* __restrict__ km, const float* __restrict__ vm, const int32_t* __restrict__ seed_idx,
                    int n_seeds, int Hq, int Hkv, int Lq, int L, int q0, int tiles, int vec,
                    float* __restrict__ out, float* __restrict__ lse) {
  using T = F32Tile<D, TM>;
  constexpr int kC = D / 32;     // output column groups of a thread (four columns each)
  extern __shared__ __align__(16) float smem[];
  float* const sq = smem;
  float* const sk = sq + T::kQ;
  float* const sv = sk + T::kKV;
  float* const sp = sv + T::kKV;
  int* const slot = reinterpret_cast<int*>(sp + T::kP);

  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  // a half-warp's 16-byte shared-memory reads merge into one access when lanes i, i ^ 1 or lanes
  // i, i ^ 2 read the same address: tx comes in adjacent pairs, tyl alternates
  const int tx = (lane >> 1) & 7, tyl = (lane & 1) | (lane >> 4) << 1;
  const int rank = C > 1 ? static_cast<int>(cluster_ctarank()) : 0;
  const unsigned unit = blockIdx.x / C;
  const unsigned head = unit / static_cast<unsigned>(tiles);        // b * Hq + hq
  const int row0 = static_cast<int>(unit - head * tiles) * T::kBM;  // first query row of the tile
  const int b = static_cast<int>(head / static_cast<unsigned>(Hq)), hq = static_cast<int>(head - b * Hq);
  const size_t kv_head = static_cast<size_t>(b) * Hkv + hq / (Hq / Hkv);
  const float* const k_base = kc + kv_head * L * D;
  const float* const v_base = vc + kv_head * L * D;
  const float scale = 1.0f / sqrtf(static_cast<float>(D));
  const int n_all = (L + kBN - 1) / kBN;
  // this CTA's key tiles (at least one: C <= n_all)
  const int j0 = C > 1 ? static_cast<int>(static_cast<long long>(rank) * n_all / C) : 0;
  const int n_kv = C > 1 ? static_cast<int>(static_cast<long long>(rank + 1) * n_all / C) : n_all;

  route_clear(slot, T::kBM, threadIdx.x, kThreads);
  griddep_wait();
  load_rows<D, T::kBM, true>(sq, q + (static_cast<size_t>(head) * Lq + row0) * D, Lq - row0, vec);
  load_rows<D, kBN, true>(sk, k_base + static_cast<size_t>(j0) * kBN * D, L - j0 * kBN, vec);
  cp_async_commit();
  load_rows<D, kBN, false>(sv, v_base + static_cast<size_t>(j0) * kBN * D, L - j0 * kBN, vec);
  cp_async_commit();
  __syncthreads();
  route_scan(slot, seed_idx + static_cast<size_t>(b) * n_seeds, n_seeds, q0 + row0, T::kBM, L, threadIdx.x, kThreads);

  const int r0 = 16 * TM / 4 * warp + tyl;   // this thread's rows are r0 + 4 i
  uint64_t o[TM][2 * kC];
  float m[TM], l[TM];
#pragma unroll
  for (int i = 0; i < TM; ++i) {
    m[i] = -INFINITY;
    l[i] = 0.0f;
#pragma unroll
    for (int c = 0; c < 2 * kC; ++c) o[i][c] = 0;
  }
  int diag[TM];   // key column of a seed row's excluded diagonal term

  for (int j = j0; j < n_kv; ++j) {
    cp_async_wait<1>();   // K(j) (and Q) have landed; V(j) may be in flight
    __syncthreads();
    if (j == j0) {
#pragma unroll
      for (int i = 0; i < TM; ++i) diag[i] = slot[r0 + 4 * i] != kNoSlot ? q0 + row0 + r0 + 4 * i : -1;
    }
    // ---- scores: partial sums over even and odd d in the two halves of a pair, and over kParts
    // stretches of d where there are registers for it (a dot product's rounding error grows with
    // its longest chain) ----
    constexpr int kParts = TM == 1 ? 4 : TM == 2 ? 2 : 1;
    float dots[TM][8];
#pragma unroll
    for (int part = 0; part < kParts; ++part) {
      uint64_t s2[TM][8];
#pragma unroll
      for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int jj = 0; jj < 8; ++jj) s2[i][jj] = 0;
#pragma unroll 4
      for (int c = part * (D / 4 / kParts); c < (part + 1) * (D / 4 / kParts); ++c) {
        ulonglong2 qa[TM];
#pragma unroll
        for (int i = 0; i < TM; ++i) {
          const int r = r0 + 4 * i;
          qa[i] = lds2(sq + r * D + 4 * (c ^ (r & 7)));
        }
        const float* kp = sk + tx * D + 4 * (c ^ tx);
#pragma unroll
        for (int jj = 0; jj < 8; ++jj) {
          const ulonglong2 ka = lds2(kp + 8 * jj * D);
#pragma unroll
          for (int i = 0; i < TM; ++i) s2[i][jj] = f2_fma(qa[i].x, ka.x, s2[i][jj]);
#pragma unroll
          for (int i = 0; i < TM; ++i) s2[i][jj] = f2_fma(qa[i].y, ka.y, s2[i][jj]);
        }
      }
#pragma unroll
      for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int jj = 0; jj < 8; ++jj) {
          float lo, hi;
          f2_unpack(s2[i][jj], lo, hi);
          dots[i][jj] = part == 0 ? lo + hi : dots[i][jj] + (lo + hi);
        }
    }
    __syncthreads();   // every warp is done with K(j)
    if (j + 1 < n_kv)
      load_rows<D, kBN, true>(sk, k_base + static_cast<size_t>(j + 1) * kBN * D, L - (j + 1) * kBN, vec);
    cp_async_commit();
    // ---- online softmax of this thread's rows; P to shared memory ----
    const int key0 = j * kBN + tx;
    // only the last tile has keys past the end, only the tiles of the diagonal an excluded key
    const bool masked = (j + 1) * kBN > L || (q0 + row0 < (j + 1) * kBN && q0 + row0 + T::kBM > j * kBN);
#pragma unroll
    for (int i = 0; i < TM; ++i) {
      float s[8], mx = -INFINITY;
#pragma unroll
      for (int jj = 0; jj < 8; ++jj) {
        const int key = key0 + 8 * jj;
        s[jj] = dots[i][jj] * scale;
        if (masked && (key >= L || key == diag[i])) s[jj] = -INFINITY;
        mx = fmaxf(mx, s[jj]);
      }
#pragma unroll
      for (int off = 8; off > 1; off >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, off));
      const float m_new = fmaxf(m[i], mx);
      const float ref = m_new == -INFINITY ? 0.0f : m_new;   // no term yet: every p is 0
      const float a = expf(m[i] - ref);
      m[i] = m_new;
      float sum = 0.0f;
      float* const pr = sp + (r0 + 4 * i) * kBN;
#pragma unroll
      for (int jj = 0; jj < 8; ++jj) {
        const float p = expf(s[jj] - ref);
        sum += p;
        const int key = tx + 8 * jj;
        pr[4 * ((key >> 2) ^ (tyl << 1)) + (key & 3)] = p;
      }
      l[i] = l[i] * a + sum;
      const uint64_t aa = f2_pack(a, a);
#pragma unroll
      for (int c = 0; c < 2 * kC; ++c) o[i][c] = f2_mul(o[i][c], aa);
    }
    cp_async_wait<1>();   // V(j) has landed; K(j + 1) may be in flight
    __syncthreads();
    // ---- O += P V ----
#pragma unroll 2
    for (int kk = 0; kk < kBN / 4; ++kk) {
      float4 pa[TM];
#pragma unroll
      for (int i = 0; i < TM; ++i)
        pa[i] = *reinterpret_cast<const float4*>(sp + (r0 + 4 * i) * kBN + 4 * (kk ^ (tyl << 1)));
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const float* vp = sv + (4 * kk + e) * D + 4 * tx;
        ulonglong2 va[kC];
#pragma unroll
        for (int c = 0; c < kC; ++c) va[c] = lds2(vp + 32 * c);
#pragma unroll
        for (int i = 0; i < TM; ++i) {
          const float p = e == 0 ? pa[i].x : e == 1 ? pa[i].y : e == 2 ? pa[i].z : pa[i].w;
          const uint64_t pp = f2_pack(p, p);
#pragma unroll
          for (int c = 0; c < kC; ++c) {
            o[i][2 * c] = f2_fma(pp, va[c].x, o[i][2 * c]);
            o[i][2 * c + 1] = f2_fma(pp, va[c].y, o[i][2 * c + 1]);
          }
        }
      }
    }
    __syncthreads();   // every warp is done with V(j)
    if (j + 1 < n_kv)
      load_rows<D, kBN, false>(sv, v_base + static_cast<size_t>(j + 1) * kBN * D, L - (j + 1) * kBN, vec);
    cp_async_commit();
  }

  bool bad = false;   // a seed row of this thread came out not finite
  if constexpr (C > 1) {
    // this split's rows to shared memory (every warp is done with K and V): O over the K tile,
    // (m, l) over the V tile
    float2* const ml = reinterpret_cast<float2*>(sv);
#pragma unroll
    for (int i = 0; i < TM; ++i) {
      const int r = r0 + 4 * i;
#pragma unroll
      for (int off = 8; off > 1; off >>= 1) l[i] += __shfl_xor_sync(0xffffffffu, l[i], off);
#pragma unroll
      for (int c = 0; c < kC; ++c)
        *reinterpret_cast<ulonglong2*>(sk + r * D + 32 * c + 4 * tx) = make_ulonglong2(o[i][2 * c], o[i][2 * c + 1]);
      if (tx == 0) ml[r] = make_float2(m[i], l[i]);
    }
    cluster_sync();
    // D / 4 lanes of a warp take a row, four columns each
    constexpr int kLanes = D / 4;
    for (int e = threadIdx.x; e < T::kBM / C * kLanes; e += kThreads) {
      const int r = e / kLanes * C + rank, c4 = e % kLanes;
      float2 st[C];
      float mm = -INFINITY;
#pragma unroll
      for (int k = 0; k < C; ++k) {
        st[k] = ld_cluster2(cluster_map(smem_u32(ml + r), k));
        mm = fmaxf(mm, st[k].x);
      }
      const int sl = slot[r];
      const bool is_seed = sl != kNoSlot;
      const size_t mrow = (kv_head * n_seeds + (is_seed ? sl : 0)) * D + 4 * c4;
      float dot = 0.0f;
      if (is_seed) {
        const float4 qv = *reinterpret_cast<const float4*>(sq + r * D + 4 * (c4 ^ (r & 7)));
        dot = fmaf(qv.x, km[mrow], fmaf(qv.y, km[mrow + 1], fmaf(qv.z, km[mrow + 2], qv.w * km[mrow + 3])));
      }
#pragma unroll
      for (int off = kLanes / 2; off > 0; off >>= 1) dot += __shfl_xor_sync(0xffffffffu, dot, off);
      const float s_self = is_seed ? dot * scale : -INFINITY;
      mm = fmaxf(mm, s_self);
      const float ref = mm == -INFINITY ? 0.0f : mm;
      float ll = 0.0f;
      float4 acc = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
#pragma unroll
      for (int k = 0; k < C; ++k) {
        const float w = expf(st[k].x - ref);
        const float4 x = ld_cluster4(cluster_map(smem_u32(sk + r * D + 4 * c4), k));
        ll = fmaf(w, st[k].y, ll);
        acc.x = fmaf(w, x.x, acc.x);
        acc.y = fmaf(w, x.y, acc.y);
        acc.z = fmaf(w, x.z, acc.z);
        acc.w = fmaf(w, x.w, acc.w);
      }
      if (is_seed) {
        // the masked-input self term (k_i, v_i)
        const float p = expf(s_self - ref);
        ll += p;
        acc.x = fmaf(p, vm[mrow], acc.x);
        acc.y = fmaf(p, vm[mrow + 1], acc.y);
        acc.z = fmaf(p, vm[mrow + 2], acc.z);
        acc.w = fmaf(p, vm[mrow + 3], acc.w);
      }
      bool redo = false;
      if (row0 + r < Lq) {
        const float inv = 1.0f / ll;
        redo = is_seed && !(isfinite(acc.x * inv) && isfinite(acc.y * inv) && isfinite(acc.z * inv) && isfinite(acc.w * inv));
        const size_t row = static_cast<size_t>(head) * Lq + row0 + r;
        float* op = out + row * D + 4 * c4;
        if (vec) {
          *reinterpret_cast<float4*>(op) = make_float4(acc.x * inv, acc.y * inv, acc.z * inv, acc.w * inv);
        } else {
          op[0] = acc.x * inv;
          op[1] = acc.y * inv;
          op[2] = acc.z * inv;
          op[3] = acc.w * inv;
        }
        if (lse != nullptr && c4 == 0) lse[row] = mm + logf(ll);
      }
      bad |= redo;
    }
    cluster_sync();   // no CTA leaves while another reads its shared memory
  } else {
#pragma unroll
    for (int i = 0; i < TM; ++i) {
      const int r = r0 + 4 * i;
#pragma unroll
      for (int off = 8; off > 1; off >>= 1) l[i] += __shfl_xor_sync(0xffffffffu, l[i], off);
      const int sl = slot[r];
      const bool warp_seed = __any_sync(0xffffffffu, sl != kNoSlot);
      if (warp_seed) {
        // merge the masked-input self term (k_i, v_i) of the warp's seed rows
        const bool is_seed = sl != kNoSlot;
        const size_t mrow = (kv_head * n_seeds + (is_seed ? sl : 0)) * D;
        float dot = 0.0f;
        if (is_seed) {
#pragma unroll
          for (int c = tx; c < D / 4; c += 8) {
            const float4 qv = *reinterpret_cast<const float4*>(sq + r * D + 4 * (c ^ (r & 7)));
            const float* kp = km + mrow + 4 * c;
            dot = fmaf(qv.x, kp[0], fmaf(qv.y, kp[1], fmaf(qv.z, kp[2], fmaf(qv.w, kp[3], dot))));
          }
        }
#pragma unroll
        for (int off = 8; off > 1; off >>= 1) dot += __shfl_xor_sync(0xffffffffu, dot, off);
        if (is_seed) {
          const float s = dot * scale;
          const float m_new = fmaxf(m[i], s);
          const float a = (m[i] == -INFINITY) ? 0.0f : expf(m[i] - m_new);
          const float p = expf(s - m_new);
          l[i] = l[i] * a + p;
          m[i] = m_new;
          const uint64_t aa = f2_pack(a, a), pp = f2_pack(p, p);
#pragma unroll
          for (int c = 0; c < kC; ++c) {
            const float* vp = vm + mrow + 32 * c + 4 * tx;
            o[i][2 * c] = f2_fma(pp, f2_pack(vp[0], vp[1]), f2_mul(o[i][2 * c], aa));
            o[i][2 * c + 1] = f2_fma(pp, f2_pack(vp[2], vp[3]), f2_mul(o[i][2 * c + 1], aa));
          }
        }
      }
      if (row0 + r < Lq) {
        const float inv = 1.0f / l[i];
        const size_t row = static_cast<size_t>(head) * Lq + row0 + r;
#pragma unroll
        for (int c = 0; c < kC; ++c) {
          float x0, x1, x2, x3;
          f2_unpack(o[i][2 * c], x0, x1);
          f2_unpack(o[i][2 * c + 1], x2, x3);
          float* op = out + row * D + 32 * c + 4 * tx;
          if (vec) {
            *reinterpret_cast<float4*>(op) = make_float4(x0 * inv, x1 * inv, x2 * inv, x3 * inv);
          } else {
            op[0] = x0 * inv;
            op[1] = x1 * inv;
            op[2] = x2 * inv;
            op[3] = x3 * inv;
          }
        }
        if (lse != nullptr && tx == 0) lse[row] = m[i] + logf(l[i]);
      }
      if (warp_seed) {
        float probe = 0.0f;   // NaN if one of this thread's sums is not finite
#pragma unroll
        for (int c = 0; c < 2 * kC; ++c) {
          float x, y;
          f2_unpack(o[i][c], x, y);
          probe = fmaf(x, 0.0f, fmaf(y, 0.0f, probe));
        }
        const bool redo = sl != kNoSlot && row0 + r < Lq && probe != 0.0f;
        bad |= redo;
      }
    }
  }
  if (__syncthreads_or(bad)) {
#pragma unroll 1
    for (int r = C > 1 ? rank + C * warp : warp; r < T::kBM && row0 + r < Lq; r += C * (kThreads / 32))
      if (slot[r] != kNoSlot)
        redo_seed_row<D>(q, kc, vc, km, vm, n_seeds, Hq, Hkv, Lq, L, q0, head, row0 + r, slot[r], out, lse);
  }
}

template <int D, int TM, int C = 1>
int launch_tile(const AttnArgs& a, bool vec, cudaStream_t stream) {
  static ContextCache<int> cache;
  int ready = 0;
  const int rc = cache.get(&ready, [](int& v) {
    v = 1;
    return cudaFuncSetAttribute(attn_f32_kernel<D, TM, C>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                static_cast<int>(F32Tile<D, TM>::kBytes)) == cudaSuccess ? 0 : -3;
  });
  if (rc != 0) return rc;
  const int tiles = (a.Lq + F32Tile<D, TM>::kBM - 1) / F32Tile<D, TM>::kBM;
  const long long blocks = static_cast<long long>(a.B) * a.Hq * tiles * C;
  if (blocks > 0x7fffffffLL) return -2;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = C;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(static_cast<unsigned>(blocks));
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = F32Tile<D, TM>::kBytes;
  cfg.stream = stream;
  cfg.attrs = attr;
  cfg.numAttrs = C > 1 ? 2 : 1;
  const cudaError_t err = cudaLaunchKernelEx(
      &cfg, attn_f32_kernel<D, TM, C>, static_cast<const float*>(a.q), static_cast<const float*>(a.k_cached),
      static_cast<const float*>(a.v_cached), static_cast<const float*>(a.k_seedmask),
      static_cast<const float*>(a.v_seedmask), a.seed_idx, a.n_seeds, a.Hq, a.Hkv, a.Lq, a.L, a.q0, tiles,
      vec ? 1 : 0, static_cast<float*>(a.out), a.lse);
  return err == cudaSuccess ? 0 : -3;
}

// Rows per CTA and key split, by the launch's predicted time. A CTA takes t us a key tile (alone on
// its SM, or less where an SM has several, which overlap) and 2 us around them; an SM with w CTAs runs
// them in w turns; combining a split costs 1 us. t as measured at D = 128 (TM = 1, 2, 4: 4.1, 5.0,
// 8.2 alone, 3.15, 4.25, 7.4 shared), about half of it at D = 64. us measured at the candidates:
//   heads x rows x keys, D      TM = 1 / 2 / 4 unsplit     TM = 1 split in 2 / 4 / 8   TM = 2 in 2 / 4
//   32 x 512 x 512, 128         177 / 136 / 119
//   8 x 512 x 512, 128          50 / 42 / 69
//   32 x 300 x 300, 128         63 / 66 / 76
//   8 x 100 x 1000, 128         65 / 80 / 131              36 / 28 / 31                44 / 24
//   2 x 1000 x 1000, 128        65                         51 / 54 / 61                44 / 39
//   4 x 256 x 256, 64           10.6 / 13.8 / 20.8         7.5 / 6.8
//   5 x 20 x 600, 64            22.4                       13.4 / 9.4 / 7.4
// Unsplit, a few rows over many keys left most SMs idle for the whole chain of key tiles.
template <int D>
int launch_rows(const AttnArgs& a, bool vec, cudaStream_t stream) {
  static ContextCache<int> cache;
  int n_sm = 0;
  const int rc = cache.get(&n_sm, [](int& v) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return -3;
    return cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess ? 0 : -3;
  });
  if (rc != 0) return rc;
  const int n_kv = (a.L + kBN - 1) / kBN;
  double best = 0.0;
  int tm = 0, split = 0;
  const auto consider = [&](int t, int c, double alone, double shared) {
    if (c > n_kv) return;
    const long long ctas = static_cast<long long>(a.B) * a.Hq * ((a.Lq + 16 * t - 1) / (16 * t)) * c;
    const long long w = (ctas + n_sm - 1) / n_sm;
    const double us = w * (2.0 + (n_kv + c - 1) / c * (w == 1 ? alone : shared) * (D == 64 ? 0.53 : 1.0)) + (c > 1);
    if (tm == 0 || us < best) best = us, tm = t, split = c;
  };
  consider(4, 1, 8.2, 7.4);
  for (const int c : {1, 2, 4}) consider(2, c, 5.0, 4.25);
  for (const int c : {1, 2, 4, 8}) consider(1, c, 4.1, 3.15);
  switch (100 * tm + split) {
    case 401: return launch_tile<D, 4>(a, vec, stream);
    case 201: return launch_tile<D, 2>(a, vec, stream);
    case 202: return launch_tile<D, 2, 2>(a, vec, stream);
    case 204: return launch_tile<D, 2, 4>(a, vec, stream);
    case 102: return launch_tile<D, 1, 2>(a, vec, stream);
    case 104: return launch_tile<D, 1, 4>(a, vec, stream);
    case 108: return launch_tile<D, 1, 8>(a, vec, stream);
    default: return launch_tile<D, 1>(a, vec, stream);
  }
}

}  // namespace

int launch_attn_f32(const AttnArgs& a, int* /*status*/, cudaStream_t stream) {
  bool vec = true;   // 16-byte copies; the entry point asks for 4-byte alignment only
  for (const void* p : {a.q, a.k_cached, a.v_cached, static_cast<const void*>(a.out)})
    vec = vec && reinterpret_cast<uintptr_t>(p) % 16 == 0;
  return a.D == 64 ? launch_rows<64>(a, vec, stream) : launch_rows<128>(a, vec, stream);
}

}  // namespace cover
