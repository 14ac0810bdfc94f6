// mass_kernel.cu - the influence terms of the seed score (Section 5.3):
//   d_in(j)  = sum over still-masked queries q of A[q -> j]
//   d_out(j) = sum over positions i drafted in this step of A[j -> i]
// with A the attention matrix of the current pass averaged over the heads,
// for the response positions pos0 .. pos0 + per - 1 of every batch row.
//
// The weights are recomputed from the attention pass's inputs and its
// log-sum-exp: A_h[q -> j] = exp(q.k'_j / sqrt(d) - lse_h(q)), where a seed
// query's diagonal entry uses its masked-input key k_q (its leave-one-out view,
// Section 5.1; the stored lse is that of the corrected distribution), so each
// row sums to one over the whole memory. Only response queries and response
// keys contribute, so the pass covers a per x per block of each head.
//
// Both sums become row sums held in registers by computing the block twice on
// the tensor cores, once per orientation, in 128 x 128 tiles:
//   row product     S  = Q_t K_j^T: thread = query row of tile t, sums its weights
//                   over the drafted keys of tile j (d_out partial);
//   column product  S' = K_t Q_j^T: thread = key of tile t, sums exp(s - lse(q)) over
//                   the masked queries q of tile j, whose lse is staged per column
//                   in shared memory (negated; -inf for a query that is not masked,
//                   so its weight is exactly 0) (d_in partial).
// A product whose tile j has no drafted key (rows) or no masked query (columns) is left out, and
// a 32-column chunk without one is skipped, as is a group of four keys without a drafted one (a step
// drafts few; the predicates are the same for every thread). Each CTA writes one partial per row of
// its tiles; a second kernel adds the partials of the Hq heads in a fixed order (deterministic) and
// divides by the head count.
//
// A CTA keeps Q_t and K_t of NT tiles of one head resident: they serve as the A operands of both
// orientations and as the B operands of the products among themselves; the block's other tiles
// stream through a two-slot ring. The math warpgroups take the products of one tile each (NT = 2,
// two warpgroups a tile, 64 columns each) or of one orientation each (NT = 1) from two tensor-memory
// buffers, so a product overlaps the previous one's exponentials.
//
// Bound: latency and, with many heads, reading Q and K once (8 x 32 heads x 256 rows: 34 MB, 5 us).
// With NT = 2 a head's 256-row block is one CTA that reads it once, instead of four CTAs (one per
// tile and orientation) reading three tiles each: 29.1 -> 17.9 us there (both launches, 32 seeds a
// sequence; 31.1 -> 19.4 with 64), 16.6 -> 9.4 us with 4 x 32 heads, 53.7 -> 34.7 us with 8 x 28/4
// heads and 512 rows. What is left is a CTA's chain in ceil(CTAs / SMs) waves, about 8 us: its tiles
// and seed keys (2 to 4 us), then four products and their exponentials. Prefetching the next wave's
// tiles and seed keys into L2 did not shorten it (19.4 us either way; 5 x 32/8, 384 rows: 23.9 -> 24.4).
//
// Warps: the math warps (thread = tensor-memory lane, a row / key of a tile), then one whose lane 0
// issues the TMA loads and one that allocates tensor memory and whose lane 0 issues the products.
#include <cuda_bf16.h>
#include <math.h>

#include "context.cuh"
#include "kernels.cuh"
#include "ptx.cuh"
#include "route.cuh"
#include "tmap.cuh"

namespace cover {
namespace {

constexpr int kD = 128;
constexpr int kT = 128;                     // rows / keys per tile
// Math warps: two warpgroups (one per tile with NT = 2, one per orientation with NT = 1); with NT = 2
// there are two of each, taking 64 of a product's 128 columns each.
template <int NT>
struct MassRoles {
  static constexpr int kHalves = NT == 2 ? 2 : 1;
  static constexpr int kMathWarps = 8 * kHalves;
  static constexpr int kTmaWarp = kMathWarps, kMmaWarp = kMathWarps + 1;
  static constexpr int kThreads = 32 * (kMathWarps + 2);
};
constexpr int kTileBytes = kT * kD * 2;     // 32 KB
constexpr int kBoxBytes = kTileBytes / 2;   // one 64-column, 128-byte-swizzled box
constexpr int kMaxPer = kMassMaxPer;        // per-column staging must fit in shared memory
constexpr int kSlots = 2;                   // ring slots of the streamed tiles
constexpr int kMaxTilesPair = 32;           // tiles of a block up to which two are resident

struct alignas(128) MassCtrl {
  uint64_t bar_q[2], bar_k[2];              // resident Q / K tile has landed
  uint64_t bar_ring_full[kSlots], bar_ring_empty[kSlots];
  uint64_t bar_s_full[2][2];                // [warpgroup][buffer]
  uint64_t bar_s_empty[2][2];
  uint64_t bar_drain;
  uint32_t tmem_base;
  int abort;
  int slot[2 * kT];                         // seed slot of the resident tiles' positions
  float half1[2][2][kT];                    // [tile][kind] sums over columns 64 .. 127 (NT = 2)
};

// Shared memory: NT Q tiles | NT K tiles | kSlots ring slots (when the block has more than NT tiles) |
// MassCtrl | per-column data of the whole block:
//   uint32_t bits[2][n_t * 4]  drafted keys, masked queries
//   float colv[n_t * 128]      the negated log2-scaled lse of a masked query, else -inf
size_t mass_smem_bytes(int NT, int n_t) {
  return static_cast<size_t>(2 * NT + (n_t > NT ? kSlots : 0)) * kTileBytes + sizeof(MassCtrl) +
         static_cast<size_t>(n_t) * (8 * sizeof(uint32_t) + kT * sizeof(float)) + 1024;
}

// blockIdx.x = (b * Hq + hq) * n_g + g: tiles NT g .. of head (b, hq).
template <int NT>
__global__ void __launch_bounds__(MassRoles<NT>::kThreads, NT == 1 ? 2 : 1)
    mass_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k,
                const __nv_bfloat16* __restrict__ k_seedmask, const int32_t* __restrict__ seed_idx, int n_seeds,
                const float* __restrict__ lse, int Hq, int Hkv, int L, int pos0, int per, int n_t, int n_g,
                const int32_t* __restrict__ tok, const uint8_t* __restrict__ flags, int mask_id, float scale_log2,
                float* __restrict__ part_in, float* __restrict__ part_out, int* status) {
  using Roles = MassRoles<NT>;
  constexpr int kTmaWarp = Roles::kTmaWarp, kMmaWarp = Roles::kMmaWarp, kThreads = Roles::kThreads;
  constexpr int kHalves = Roles::kHalves;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* const base =
      reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* const xq = base;
  uint8_t* const xk = base + NT * kTileBytes;
  uint8_t* const ring = base + 2 * NT * kTileBytes;
  MassCtrl& sm = *reinterpret_cast<MassCtrl*>(ring + (n_t > NT ? kSlots * kTileBytes : 0));
  uint32_t* const bits = reinterpret_cast<uint32_t*>(&sm + 1);   // [kind][n_t * 4]
  float* const colv = reinterpret_cast<float*>(bits + 8 * n_t);

  const int tid = threadIdx.x;
  const int warp = tid >> 5, lane = tid & 31;
  const int bh = static_cast<int>(blockIdx.x) / n_g;   // b * Hq + hq
  const int t0 = (static_cast<int>(blockIdx.x) - bh * n_g) * NT;
  const int nw = min(NT, n_t - t0);                    // resident tiles
  const int hq = bh % Hq, b = bh / Hq;
  const int hkv = hq / (Hq / Hkv);
  // tensor-memory buffers of a warpgroup (one for a one-tile block, so that two CTAs share an SM)
  const int nbuf = n_t == 1 ? 1 : 2;
  const uint32_t tmem_cols = 2u * static_cast<uint32_t>(nbuf) * kT;
  // the block's tiles in the order they are taken: the resident ones first
  auto tile_of = [&](int jj) {
    if (jj < nw) return t0 + jj;
    const int o = jj - nw;
    return o < t0 ? o : o + nw;
  };
  // whether tile j has a drafted key (kind 0, row products) / a masked query (kind 1, column products)
  auto needed = [&](int kind, int j) {
    const uint4 w = reinterpret_cast<const uint4*>(bits + kind * 4 * n_t)[j];
    return (w.x | w.y | w.z | w.w) != 0u;
  };

  if (warp == kTmaWarp && lane == 0) {
    for (int s = 0; s < 2; ++s) {
      mbar_init(&sm.bar_q[s], 1);
      mbar_init(&sm.bar_k[s], 1);
      mbar_init(&sm.bar_ring_full[s], 1);
      mbar_init(&sm.bar_ring_empty[s], 1);
      for (int u = 0; u < 2; ++u) {
        mbar_init(&sm.bar_s_full[s][u], 1);
        mbar_init(&sm.bar_s_empty[s][u], 4 * kHalves);
      }
    }
    mbar_init(&sm.bar_drain, 1);
    sm.abort = 0;
    fence_mbar_init();
    tma_prefetch_desc(&tm_q);
    tma_prefetch_desc(&tm_k);
  }
  if (warp == kMmaWarp) {
    tmem_alloc(&sm.tmem_base, tmem_cols);
    tmem_relinquish();
  }
  route_clear(sm.slot, 2 * kT, tid, kThreads);
  // launched as a programmatic dependent of the stream's previous kernel: wait for its results;
  // the reduction kernel behind this one may be scheduled now, it waits for this grid's results
  griddep_wait();
  griddep_launch_dependents();
  if (warp == kTmaWarp && lane == 0) {
    // the resident tiles are issued at once, so their latency overlaps the rest of the prologue
    for (int w = 0; w < nw; ++w)
      for (int kind = 0; kind < 2; ++kind) {
        uint64_t* bar = kind == 0 ? &sm.bar_q[w] : &sm.bar_k[w];
        mbar_arrive_expect_tx(bar, kTileBytes);
        for (int h = 0; h < 2; ++h)
          tma_load_4d((kind == 0 ? xq : xk) + w * kTileBytes + h * kBoxBytes, kind == 0 ? &tm_q : &tm_k, bar, 64 * h,
                      pos0 + (t0 + w) * kT, kind == 0 ? hq : hkv, b);
      }
  }
  // the first seed entry of this thread, loaded now so that its latency overlaps the column data's
  const int32_t* seeds_b = seed_idx + static_cast<size_t>(b) * n_seeds;
  const int seed0 = tid < n_seeds ? __ldg(seeds_b + tid) : -1;
  // per-column data of the whole block: the drafted keys, the masked queries and their lse; one
  // warp per 32 columns
  for (int w = warp; w < n_t * 4; w += kThreads / 32) {
    const int c = w * 32 + lane;
    const bool in = c < per;
    const size_t srow = static_cast<size_t>(b) * per + c;
    const bool drafted = in && (flags[srow] & 2u) != 0;
    const bool masked = in && tok[srow] == mask_id;
    const float l2 = in ? lse[static_cast<size_t>(bh) * L + pos0 + c] * 1.4426950408889634f : 0.0f;
    colv[c] = masked ? -l2 : -INFINITY;
    const uint32_t d = __ballot_sync(0xffffffffu, drafted), m = __ballot_sync(0xffffffffu, masked);
    if (lane == 0) {
      bits[w] = d;
      bits[4 * n_t + w] = m;
    }
  }
  // the log2-scaled lse of a math thread's own query (thread = row of its tile)
  const int g = (warp >> 2) & 1;                       // tile (NT = 2) or orientation (NT = 1) of its products
  const int half = warp >> 3;                          // and the 64 columns it takes of them (NT = 2)
  const int my = NT == 2 ? g : 0;                      // its resident tile
  const int r = tid & (kT - 1);                        // tensor-memory lane
  const int i = (t0 + my) * kT + r;                    // response index of this thread's query / key
  const bool valid = warp < Roles::kMathWarps && my < nw && i < per;
  const float own = valid ? lse[static_cast<size_t>(bh) * L + pos0 + i] * 1.4426950408889634f : 0.0f;
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  {
    // seed routing of the resident tiles' positions (the lowest slot naming a position wins)
    const int row0 = pos0 + t0 * kT, rows = nw * kT;
    if (seed0 >= row0 && seed0 < row0 + rows && seed0 < L) atomicMin(sm.slot + (seed0 - row0), tid);
    for (int sidx = tid + kThreads; sidx < n_seeds; sidx += kThreads) {
      const int p = __ldg(seeds_b + sidx);
      if (p >= row0 && p < row0 + rows && p < L) atomicMin(sm.slot + (p - row0), sidx);
    }
  }
  __syncthreads();
  const uint32_t tbase = sm.tmem_base;
  float sum[2] = {0.0f, 0.0f};   // NT = 2: this thread's sums over its half of the columns
  bool done = false;             // and whether it adds the other half's and writes them

  if (warp == kTmaWarp) {
    if (lane == 0) {
      int n = 0;   // tiles streamed so far
      bool ok = true;
      for (int jj = nw; jj < n_t && ok; ++jj) {
        const int j = tile_of(jj);
        for (int kind = 0; kind < 2 && ok; ++kind) {
          if (!needed(kind, j)) continue;
          // a row product streams K_j, a column product Q_j
          const int st = n % kSlots, use = n / kSlots;
          ok = use == 0 || mbar_wait(&sm.bar_ring_empty[st], (use - 1) & 1, &sm.abort);
          if (!ok) break;
          mbar_arrive_expect_tx(&sm.bar_ring_full[st], kTileBytes);
          for (int h = 0; h < 2; ++h)
            tma_load_4d(ring + st * kTileBytes + h * kBoxBytes, kind == 0 ? &tm_k : &tm_q, &sm.bar_ring_full[st],
                        64 * h, pos0 + j * kT, kind == 0 ? hkv : hq, b);
          ++n;
        }
      }
      if (!ok) {
        report_status(status, kStatusTimeout, 60);
        sm.abort = 1;
      }
      // let every copy issued land before the CTA's shared memory is released: the resident tiles
      // whose products were left out, the rest on an abort
      for (int w = 0; w < nw; ++w) {
        mbar_wait(&sm.bar_q[w], 0, nullptr);
        mbar_wait(&sm.bar_k[w], 0, nullptr);
      }
      for (int e = max(0, n - kSlots); e < n; ++e) mbar_wait(&sm.bar_ring_full[e % kSlots], (e / kSlots) & 1, nullptr);
    }
  } else if (warp == kMmaWarp) {
    if (lane == 0) {
      constexpr uint32_t id_s = idesc_bf16_f32(kT, kT, false, false);
      constexpr uint64_t kTileDesc = kTileBytes >> 4;
      const uint64_t dq = sdesc_sw128(smem_u32(xq), 16, 1024);
      const uint64_t dk = sdesc_sw128(smem_u32(xk), 16, 1024);
      const uint64_t dr = sdesc_sw128(smem_u32(ring), 16, 1024);
      int n = 0;              // streamed tiles taken
      int k[2] = {0, 0};      // products issued to each warpgroup
      bool ok = true;
      for (int jj = 0; jj < n_t && ok; ++jj) {
        const int j = tile_of(jj);
        for (int kind = 0; kind < 2 && ok; ++kind) {
          if (!needed(kind, j)) continue;
          // B: K_j (rows) or Q_j (columns), resident or streamed
          uint64_t db;
          if (jj < nw) {
            ok = mbar_wait(kind == 0 ? &sm.bar_k[jj] : &sm.bar_q[jj], 0, &sm.abort);
            db = (kind == 0 ? dk : dq) + jj * kTileDesc;
          } else {
            ok = mbar_wait(&sm.bar_ring_full[n % kSlots], (n / kSlots) & 1, &sm.abort);
            db = dr + (n % kSlots) * kTileDesc;
          }
          for (int w = 0; w < nw && ok; ++w) {
            const int wg = NT == 2 ? w : kind;
            const int buf = k[wg] % nbuf, use = k[wg] / nbuf;
            ok = mbar_wait(kind == 0 ? &sm.bar_q[w] : &sm.bar_k[w], 0, &sm.abort) &&
                 (use == 0 || mbar_wait(&sm.bar_s_empty[wg][buf], (use - 1) & 1, &sm.abort));
            if (!ok) break;
            tc_fence_after_sync();
            // S = A . B^T, both K-major with 128-byte swizzle
            const uint64_t da = (kind == 0 ? dq : dk) + w * kTileDesc;
#pragma unroll
            for (int ks = 0; ks < kD / 16; ++ks) {
              const uint64_t off = static_cast<uint64_t>(((ks >> 2) * kBoxBytes + (ks & 3) * 32) >> 4);
              umma_ss(tbase + (wg * nbuf + buf) * kT, da + off, db + off, id_s, ks > 0 ? 1u : 0u);
            }
            umma_commit(&sm.bar_s_full[wg][buf]);
            ++k[wg];
          }
          if (jj >= nw) {
            umma_commit(&sm.bar_ring_empty[n % kSlots]);
            ++n;
          }
        }
      }
      if (!ok) {
        report_status(status, kStatusTimeout, 61);
        sm.abort = 1;
      }
      // all tensor-core work of this CTA must finish before tensor memory is released
      umma_commit(&sm.bar_drain);
      mbar_wait(&sm.bar_drain, 0, nullptr);
    }
  } else if (my < nw) {
    // ---------------- rows / keys of the resident tiles ----------------
    const uint32_t trow = tbase + (static_cast<uint32_t>((warp & 3) * 32) << 16);
    // the diagonal entry of a seed query uses its masked-input key (leave-one-out view): its score
    // replaces the cached one before the exponentials
    // (in the half of the columns that holds the diagonal)
    const int my_slot = valid && (kHalves == 1 || r / 64 == half) ? sm.slot[my * kT + r] : kNoSlot;
    uint32_t pending = __ballot_sync(0xffffffffu, my_slot != kNoSlot);
    const bool warp_seed = pending != 0u;
    float s_self = 0.0f;
    bool ok = true;
    if (warp_seed) {
      // four seed rows at a time, eight lanes each (lane l of the eight takes dimensions 16 l .. + 15),
      // the next four rows' keys on their way; the first ones' are, while the Q tile lands
      const __nv_bfloat16* km = k_seedmask + (static_cast<size_t>(b) * Hkv + hkv) * n_seeds * kD;
      const int gl = lane & 7;
      int src = -1;
      uint4 kv[2];
      const auto fetch = [&] {
        uint32_t p = pending;
        for (int e = lane >> 3; e > 0; --e) p &= p - 1u;
        src = p != 0u ? __ffs(p) - 1 : -1;
        const int sl = __shfl_sync(0xffffffffu, my_slot, src & 31);
        if (src >= 0) {
          const uint4* krow = reinterpret_cast<const uint4*>(km + static_cast<size_t>(sl) * kD) + 2 * gl;
          kv[0] = __ldg(krow);
          kv[1] = __ldg(krow + 1);
        }
      };
      fetch();
      ok = __all_sync(0xffffffffu, mbar_wait(&sm.bar_q[my], 0, &sm.abort));
      const uint8_t* qbox = xq + my * kTileBytes + (gl >> 2) * kBoxBytes;
#pragma unroll 1
      while (ok && pending != 0u) {
        const int from = src;
        const uint4 k0 = kv[0], k1 = kv[1];
#pragma unroll
        for (int e = 0; e < 4; ++e) pending &= pending - 1u;
        if (pending != 0u) fetch();
        const int row = (warp & 3) * 32 + (from & 31);
        float dot = 0.0f;
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          const uint4 qv = *reinterpret_cast<const uint4*>(qbox + row * 128 + (((2 * (gl & 3) + c) ^ (row & 7)) << 4));
          const __nv_bfloat162* qp = reinterpret_cast<const __nv_bfloat162*>(&qv);
          const __nv_bfloat162* kp = reinterpret_cast<const __nv_bfloat162*>(c == 0 ? &k0 : &k1);
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const float2 qf = __bfloat1622float2(qp[e]), kf = __bfloat1622float2(kp[e]);
            dot = fmaf(qf.x, kf.x, fmaf(qf.y, kf.y, dot));
          }
        }
#pragma unroll
        for (int o = 4; o >= 1; o >>= 1) dot += __shfl_xor_sync(0xffffffffu, dot, o);
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const int at = __shfl_sync(0xffffffffu, from, 8 * e);
          const float v = __shfl_sync(0xffffffffu, dot, 8 * e);
          if (lane == at) s_self = v;
        }
      }
    }
    const uint64_t scale2 = f2_pack(scale_log2, scale_log2), nown2 = f2_pack(-own, -own);
    float acc[2] = {0.0f, 0.0f};   // rows, columns
    int k = 0;
    for (int jj = 0; jj < n_t && ok; ++jj) {
      const int j = tile_of(jj);
#pragma unroll
      for (int kind = 0; kind < 2; ++kind) {
        if (!needed(kind, j) || (NT == 1 && kind != g) || !ok) continue;
        const int buf = k % nbuf;
        ok = __all_sync(0xffffffffu, mbar_wait(&sm.bar_s_full[g][buf], (k / nbuf) & 1, &sm.abort));
        if (!ok) break;
        ++k;
        tc_fence_after_sync();
        const int diag = my_slot != kNoSlot ? r : -1;   // column of the seed diagonal in tile t0 + my
        uint64_t a2[2] = {0, 0};
        // a quarter of the tile at a time, in a rolled loop: a CTA runs through its code once or
        // twice, and what it has to fetch counts
        constexpr int kQuarters = 4 / kHalves;
        const int q0 = kHalves == 2 ? 2 * half : 0;
#pragma unroll 1
        for (int c32 = q0; c32 < q0 + kQuarters; ++c32) {
          const uint32_t word = bits[(kind * n_t + j) * 4 + c32];   // the same for every thread
          uint32_t raw[32];
          if (word != 0u) {
            tmem_ld32(trow + (g * nbuf + buf) * kT + 32 * c32, raw);
            tmem_ld_wait(raw);
          }
          if (c32 == q0 + kQuarters - 1) {
            tc_fence_before_sync();
            __syncwarp();
            if (lane == 0) mbar_arrive(&sm.bar_s_empty[g][buf]);
          }
          if (word == 0u) continue;
          float* s = reinterpret_cast<float*>(raw);
          if (warp_seed && j == t0 + my) {
#pragma unroll
            for (int c = 0; c < 32; ++c)
              if (32 * c32 + c == diag) s[c] = s_self;
          }
#pragma unroll
          for (int e4 = 0; e4 < 8; ++e4) {
            const uint32_t nib = (word >> (4 * e4)) & 15u;
            if (kind == 0 && nib == 0u) continue;
            const float* s4 = s + 4 * e4;
            float p[4];
            if (kind == 0) {
#pragma unroll
              for (int e = 0; e < 4; e += 2) {
                float x, y;
                f2_unpack(f2_fma(f2_pack(s4[e], s4[e + 1]), scale2, nown2), x, y);
                p[e] = (nib >> e) & 1u ? ex2_approx(x) : 0.0f;
                p[e + 1] = (nib >> (e + 1)) & 1u ? ex2_approx(y) : 0.0f;
              }
            } else {
              // the queries' negated lse, -inf where not masked (weight 0)
              const float4 v = *reinterpret_cast<const float4*>(colv + j * kT + 32 * c32 + 4 * e4);
              float x, y;
              f2_unpack(f2_fma(f2_pack(s4[0], s4[1]), scale2, f2_pack(v.x, v.y)), x, y);
              p[0] = ex2_approx(x);
              p[1] = ex2_approx(y);
              f2_unpack(f2_fma(f2_pack(s4[2], s4[3]), scale2, f2_pack(v.z, v.w)), x, y);
              p[2] = ex2_approx(x);
              p[3] = ex2_approx(y);
            }
            a2[0] = f2_add(a2[0], f2_pack(p[0], p[1]));
            a2[1] = f2_add(a2[1], f2_pack(p[2], p[3]));
          }
        }
        float a4[4];
        f2_unpack(a2[0], a4[0], a4[1]);
        f2_unpack(a2[1], a4[2], a4[3]);
        acc[kind] += (a4[0] + a4[1]) + (a4[2] + a4[3]);
      }
    }
    if (!ok) {
      if (lane == 0 && !sm.abort) {
        report_status(status, kStatusTimeout, 62);
        sm.abort = 1;
      }
    } else if (kHalves == 2) {
      if (half == 1) {
        sm.half1[my][0][r] = acc[0];
        sm.half1[my][1][r] = acc[1];
      }
      sum[0] = acc[0];
      sum[1] = acc[1];
      done = valid && half == 0;
    } else if (valid) {
      const size_t o = static_cast<size_t>(bh) * per + i;
      if (g == 0) part_out[o] = acc[0];
      else part_in[o] = acc[1];
    }
  }

  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  if (kHalves == 2 && done) {
    const size_t o = static_cast<size_t>(bh) * per + i;
    part_out[o] = sum[0] + sm.half1[my][0][r];
    part_in[o] = sum[1] + sm.half1[my][1][r];
  }
  if (warp == kMmaWarp) tmem_dealloc(tbase, tmem_cols);
}

// d_in / d_out of row n = b * per + i: the partial sums of the Hq heads in a fixed order, divided
// by the head count. A CTA takes 32 rows; warp w adds heads w, w + 8, ..., then the eight sums are
// added in order (one thread per row walking all heads was a chain of Hq loads).
constexpr int kReduceWarps = 8;
__global__ void __launch_bounds__(32 * kReduceWarps)
    mass_reduce_kernel(const float* __restrict__ part_in, const float* __restrict__ part_out, int B, int Hq, int per,
                       float* __restrict__ d_in, float* __restrict__ d_out) {
  __shared__ float sums[2][kReduceWarps][32];
  // launched as a programmatic dependent of mass_kernel: wait until its partial sums are complete
  // and visible
  griddep_wait();
  griddep_launch_dependents();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int n = blockIdx.x * 32 + lane;
  const bool in = n < B * per;
  const int b = in ? n / per : 0, i = in ? n - b * per : 0;
  float si = 0.0f, so = 0.0f;
#pragma unroll 4
  for (int h = warp; h < Hq; h += kReduceWarps) {
    const size_t o = (static_cast<size_t>(b) * Hq + h) * per + i;
    si += part_in[o];
    so += part_out[o];
  }
  sums[0][warp][lane] = si;
  sums[1][warp][lane] = so;
  __syncthreads();
  if (warp < 2 && in) {
    float t = sums[warp][0][lane];
#pragma unroll
    for (int w = 1; w < kReduceWarps; ++w) t += sums[warp][w][lane];
    (warp == 0 ? d_in : d_out)[n] = t * (1.0f / static_cast<float>(Hq));
  }
}

template <int NT>
int launch_tiles(const MassArgs& a, int n_t, const CUtensorMap& tq, const CUtensorMap& tk, float* part_in,
                 float* part_out, int* status, cudaStream_t stream) {
  // the shared-memory limit is a function attribute of the current context
  static ContextCache<int> setup;
  int unused = 0;
  const int rc = setup.get(&unused, [](int&) {
    const size_t most = mass_smem_bytes(NT, NT == 2 ? kMaxTilesPair : (kMaxPer + kT - 1) / kT);
    return cudaFuncSetAttribute(mass_kernel<NT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                static_cast<int>(most)) == cudaSuccess ? 0 : -3;
  });
  if (rc != 0) return rc;
  const int n_g = (n_t + NT - 1) / NT;
  const long long grid = static_cast<long long>(n_g) * a.Hq * a.B;
  if (grid > 0x7fffffffLL) return -2;
  const float scale_log2 = 1.4426950408889634f / sqrtf(static_cast<float>(kD));
  cudaLaunchAttribute attr[1];
  const cudaLaunchConfig_t cfg =
      pdl_config(dim3(static_cast<unsigned>(grid)), dim3(MassRoles<NT>::kThreads), mass_smem_bytes(NT, n_t), stream,
                 attr);
  return cudaLaunchKernelEx(&cfg, mass_kernel<NT>, tq, tk, static_cast<const __nv_bfloat16*>(a.k_seedmask), a.seed_idx,
                            a.n_seeds, a.lse, a.Hq, a.Hkv, a.L, a.pos0, a.per, n_t, n_g, a.tok, a.flags, a.mask_id,
                            scale_log2, part_in, part_out, status) == cudaSuccess ? 0 : -3;
}

}  // namespace

size_t mass_workspace_bytes(int B, int Hq, int per) {
  return 2 * sizeof(float) * static_cast<size_t>(B) * Hq * per;
}

int launch_attn_mass(const MassArgs& a, int* status, cudaStream_t stream) {
  if (a.per > kMaxPer) return -2;
  CUtensorMap tq, tk;
  if (!make_bf16_map_4d(&tq, a.q, kD, a.L, a.Hq, a.B, kT) || !make_bf16_map_4d(&tk, a.k_cached, kD, a.L, a.Hkv, a.B, kT))
    return -3;
  const int n_t = (a.per + kT - 1) / kT;
  if (static_cast<long long>(n_t) * a.Hq * a.B > 0x7fffffffLL) return -2;
  float* part_in = static_cast<float*>(a.workspace);
  float* part_out = part_in + static_cast<size_t>(a.B) * a.Hq * a.per;
  static ContextCache<int> sms;
  int n_sm = 0;
  int rc = sms.get(&n_sm, [](int& v) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return -3;
    return cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess ? 0 : -3;
  });
  if (rc != 0) return rc;
  // Tiles per CTA: two while the tiles outnumber the SMs; below that one tile a CTA spreads over
  // more SMs. us at NT = 1 / 2, 32 seeds (B, heads, rows: tiles), both launches: 1, 32, 256: 64 8.1 / 8.6;
  // 1, 28/4, 512: 112 11.2 / 12.3; 2, 28/4, 256: 112 9.2 / 8.9; 2, 32/8, 256: 128 8.4 / 9.0; 1, 32/8, 512: 128
  // 10.5 / 11.9; 2, 38, 256: 152 9.5 / 9.4; 1, 32, 640: 160 21.1 / 13.8; 3, 28/4, 256: 168 14.3 / 9.5; 4, 32,
  // 256: 256 14.6 / 9.5; 1, 32, 1024: 256 30.1 / 18.5.
  const bool pair = n_t > 1 && n_t <= kMaxTilesPair && static_cast<long long>(n_t) * a.Hq * a.B > n_sm;
  rc = pair ? launch_tiles<2>(a, n_t, tq, tk, part_in, part_out, status, stream)
            : launch_tiles<1>(a, n_t, tq, tk, part_in, part_out, status, stream);
  if (rc != 0) return rc;
  // the reduction may launch while the partial sums are still being written (programmatic
  // dependent launch); it waits on the device for them, so its launch latency is hidden
  const int rows = a.B * a.per;
  cudaLaunchAttribute attr[1];
  const cudaLaunchConfig_t cfg = pdl_config(dim3(static_cast<unsigned>((rows + 31) / 32)), dim3(32 * kReduceWarps), 0, stream, attr);
  return cudaLaunchKernelEx(&cfg, mass_reduce_kernel, static_cast<const float*>(part_in),
                            static_cast<const float*>(part_out), a.B, a.Hq, a.per, a.d_in, a.d_out) == cudaSuccess
             ? 0 : -3;
}

}  // namespace cover
