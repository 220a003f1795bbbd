// The parts of the prefill kernels (prefill_tc.cu: a CTA an item, or half of one;
// prefill_short.cu: one pipeline through many short items): shapes, the geometry of
// a work item and its copies, the MMAs and the softmax of one tile, and the output
// rows.
#pragma once

#include <math.h>

#include "common.cuh"
#include "internal.h"
#include "tc.cuh"

namespace aoh {
namespace pf {

using bf16 = __nv_bfloat16;
constexpr int kBM = 128;         // rows per query tile (a CTA owns two)
constexpr int kBN = 128;         // keys per KV tile
constexpr int kNS = 4;           // KV ring stages (K and V tiles alternate)
constexpr float kRescaleThreshold = 8.0f;
constexpr uint32_t kTmemCols = 512;
constexpr int kThreads = 320;

template <int D>
struct PfCfg {
  static constexpr int DBLK = D / 64;            // 64-wide column blocks (one TMA box each)
  static constexpr int BOX = 128 * 64 * 2;       // bytes of one [128 rows][64] box
  static constexpr int QBYTES = DBLK * BOX;      // one query tile
  static constexpr int KVBYTES = DBLK * BOX;
  static constexpr int OFF_Q = 0;                // Q_A, Q_B
  static constexpr int OFF_KV = OFF_Q + 2 * QBYTES;
  static constexpr int OFF_BAR = OFF_KV + kNS * KVBYTES;
  static constexpr int NBAR = 1 + 2 * kNS + 2 + 4 + 2 + 1 + 2;
  static constexpr int SMEM = OFF_BAR + NBAR * 8 + 16 + 1024;
  static constexpr uint32_t IDESC_S = idesc_bf16(kBM, kBN, false);
  static constexpr uint32_t IDESC_PV = idesc_bf16(kBM, D, true);
  static_assert(SMEM <= 232448, "shared memory");
  static_assert(256 + 2 * D <= (int)kTmemCols, "TMEM columns");
  static_assert(128 * (D * 4 + 8) <= OFF_BAR - QBYTES, "receive buffer of the split and its output rows");
};

// Bits lo..hi-1 of a 32-bit word (lo, hi clamped to [0, 32]).
__device__ __forceinline__ uint32_t range_bits(int lo, int hi) {
  lo = max(lo, 0);
  hi = min(hi, 32);
  if (hi <= lo) return 0u;
  const uint32_t top = hi == 32 ? 0xffffffffu : ((1u << hi) - 1u);
  return top & ~((1u << lo) - 1u);
}

// CAP: the work items that travel as arguments at most (0: they are in a.work).
template <int CAP>
struct WorkList {
  uint64_t item[CAP > 0 ? CAP : 1];
};

// A work item: two query tiles of sequence b, 0 and 1 (A and B), and the KV tiles
// they visit: the n_c tiles of cached rows, then chunk tiles [0, a_end)
// and [c_begin, c_end). Rows q0 .. q0 + 127 of heads h and h + 1, or rows q0 ..
// q0 + 255 of head h.
struct Item {
  int b, h, kvh, q0, len, Lb, S_rel, n_c, a_end, c_begin, c_end;
  bool streaming, two_heads;
  __device__ __forceinline__ Item(const PrefillTcArgs& a, uint64_t code) {
    const CacheGeom& g = a.geom;
    two_heads = (code & kPrefillTwoHeads) != 0;
    code &= ~kPrefillTwoHeads;
    b = (int)(code >> 34);
    h = (int)(code >> 24) & 1023;
    q0 = (int)(code & 0xffffffu) * (two_heads ? kBM : 2 * kBM);
    kvh = h / g.G;
    streaming = g.kind[kvh] != 0;
    const int2 chunk = a.chunk.of(b);
    len = chunk.x;
    Lb = chunk.y;
    const int q_end = min(q0 + (two_heads ? kBM : 2 * kBM), len);
    S_rel = g.S - Lb;
    n_c = Lb == 0 ? 0 : ((streaming ? min(Lb, g.S + g.W) : Lb) + kBN - 1) / kBN;
    if (!streaming) {
      a_end = (q_end + kBN - 1) / kBN;
      c_begin = c_end = a_end;
    } else {
      a_end = (min(max(S_rel, 0), q_end) + kBN - 1) / kBN;
      c_begin = max(a_end, max(0, g.wstart(q0)) / kBN);
      c_end = max(c_begin, (q_end + kBN - 1) / kBN);
    }
  }
  // query tile x: its first row and its head
  __device__ __forceinline__ int row0(int x) const { return two_heads ? q0 : q0 + x * kBM; }
  __device__ __forceinline__ int head(int x) const { return two_heads ? h + x : h; }
  __device__ __forceinline__ int tiles() const { return n_c + a_end + (c_end - c_begin); }
  // visited tile i: the chunk tile, for i >= n_c
  __device__ __forceinline__ int chunk_tile(int i) const { return i - n_c < a_end ? i - n_c : c_begin + (i - n_c - a_end); }
  // keys of visited tile i that hold data (the rest: cache rows not yet written,
  // or chunk padding); fewer than kBN makes the tile partial
  __device__ __forceinline__ int valid(const CacheGeom& g, int i) const {
    if (i < n_c) return (streaming ? min(Lb, g.S + g.W) : Lb) - i * kBN;
    return len - chunk_tile(i) * kBN;
  }
};

// TMA of visited tile i's K (sel 0) or V (sel 1) into dst; one thread.
template <int D>
__device__ __forceinline__ void load_kv(const PrefillTcArgs& a, const Item& t, int i, int sel, uint8_t* dst,
                                        uint64_t* bar) {
  using C = PfCfg<D>;
  mbar_arrive_expect_tx(bar, C::KVBYTES);
  if (i < t.n_c) {
    // cache region viewed as [regions][K, V][rows][D]
    const CacheGeom& g = a.geom;
    const CUtensorMap* map = t.streaming ? &a.tcs : &a.tcr;
    const int region = t.streaming ? t.b * g.n_s + g.idx[t.kvh] : t.b * g.n_r + g.idx[t.kvh];
    for (int db = 0; db < C::DBLK; ++db) tma_load_4d(dst + db * C::BOX, map, db * 64, i * kBN, sel, region, bar);
  } else {
    const CUtensorMap* map = sel ? &a.tv : &a.tk;
    for (int db = 0; db < C::DBLK; ++db) tma_load_4d(dst + db * C::BOX, map, db * 64, t.kvh, t.chunk_tile(i) * kBN, t.b, bar);
  }
}

// Query tile x (0: A, 1: B) of an item; one thread.
template <int D>
__device__ __forceinline__ void load_q(const PrefillTcArgs& a, const Item& t, int x, uint8_t* dst, uint64_t* bar) {
  using C = PfCfg<D>;
  mbar_arrive_expect_tx(bar, C::QBYTES);
  for (int db = 0; db < C::DBLK; ++db)
    tma_load_4d(dst + db * C::BOX, &a.tq, db * 64, t.head(x), t.row0(x), t.b, bar);
}

// Zero the rows of a landed V tile past its valid keys; one warp.
template <int D>
__device__ __forceinline__ void zero_tail(uint8_t* vt, int valid, int lane) {
  using C = PfCfg<D>;
  for (int idx = max(valid, 0) * 8 + lane; idx < kBN * 8; idx += 32) {  // 16-byte chunks
    const int row = idx >> 3, chunk = idx & 7;
#pragma unroll
    for (int db = 0; db < C::DBLK; ++db)
      *reinterpret_cast<uint4*>(vt + db * C::BOX + row * 128 + chunk * 16) = make_uint4(0, 0, 0, 0);
  }
  fence_proxy_async_smem();
  __syncwarp();
}

// S_X = Q_X K^T; one thread. q_desc, k_desc: descriptors of the query tile and of
// the K tile.
template <int D>
__device__ __forceinline__ void issue_s(uint32_t tmem, uint64_t q_desc, uint64_t k_desc, int x) {
  using C = PfCfg<D>;
#pragma unroll
  for (int kk = 0; kk < D / 16; ++kk) {
    const uint32_t off = sdesc_step((kk >> 2) * C::BOX + (kk & 3) * 32);
    tc_mma(tmem + x * 128, q_desc + off, k_desc + off, C::IDESC_S, kk > 0 ? 1u : 0u);
  }
}

// O_X (+)= P_X V over half of the tile's keys (0-63 or 64-127); one thread.
// v_desc: descriptor of the V tile.
template <int D>
__device__ __forceinline__ void issue_pv(uint32_t tmem, uint64_t v_desc, int x, int half, bool first) {
  using C = PfCfg<D>;
#pragma unroll
  for (int k = 0; k < kBN / 32; ++k) {
    const int kk = half * (kBN / 32) + k;
    tc_mma_ts(tmem + 256 + x * D, tmem + x * 128 + kk * 8, v_desc + sdesc_step(kk * 16 * 128), C::IDESC_PV,
              (kk > 0 || !first) ? 1u : 0u);
  }
}

// The keys of a visited tile that a row sees, in tile coordinates: [0, e_hi),
// [a0, a1) and [b0, b1); need = false: all. It depends on positions alone and is
// formed before the wait for S, whose end starts the loop's critical path.
struct Mask {
  bool need;
  int e_hi = kBN, a0 = 0, a1 = 0, b0 = 0, b1 = 0;
  // ja: the visited tile, i: the row's position in the chunk, qx0: the query
  // tile's first row, rot: oldest ring slot of a wrapped cached ring
  __device__ __forceinline__ Mask(const CacheGeom& g, const Item& t, int ja, int i, int qx0, int rot) {
    const int S = g.S, W = g.W, Lb = t.Lb, len = t.len, S_rel = t.S_rel;
    const int j0 = (ja < t.n_c ? ja : t.chunk_tile(ja)) * kBN;
    if (ja < t.n_c) {
      if (!t.streaming) {
        need = j0 + kBN > Lb;
        e_hi = Lb - j0;
      } else {
        need = true;
        e_hi = min(S, Lb) - j0;
        // cached positions the row may see: sinks, and [Lb + wstart(i), Lb)
        const int skip = W + g.wstart(i);  // oldest ring positions hidden
        if (Lb <= S + W) {
          a0 = max(S, Lb + g.wstart(i)) - j0;
          a1 = Lb - j0;
        } else if (skip < W) {
          const int u = rot + max(skip, 0);
          if (u < W) {
            a0 = S + u - j0;
            a1 = S + W - j0;
            b0 = S - j0;
            b1 = S + rot - j0;
          } else {
            a0 = S + u - W - j0;
            a1 = S + rot - j0;
          }
        }
      }
    } else {
      const int jl = j0 + kBN - 1;
      need = !(jl <= qx0 && jl < len && (!t.streaming || jl < S_rel || j0 >= g.wstart(qx0 + kBM - 1)));
      const int kmax = min(i, len - 1) - j0;
      if (!t.streaming) {
        e_hi = kmax + 1;
      } else {
        e_hi = min(kmax + 1, S_rel - j0);
        a0 = g.wstart(i) - j0;
        a1 = kmax + 1;
      }
    }
  }
};

// The softmax of one landed S tile, one row (TMEM lane) a thread: reads the row,
// hides keys, moves the running max m (rescaling O in TMEM when it grew by more
// than 2^8, once the PV before, phase pv_parity of pv_done, has landed), writes P
// over S's first 64 columns, announcing its two halves on p_full[0] and [1], and
// adds to l. first: no PV of this query tile before. Returns false when a wait
// gave up (uniform over the warp).
//
// The time from S to P bounds the main loop: the tensor pipe has 2048 clocks of
// work for a pair of tiles, and each of the two softmaxes has to end within the
// other's MMAs. Announcing P in halves lets P V start on keys 0-63 while the
// last quarter's weights are formed, and the mask's key ranges are known before S
// lands: 32K causal tokens of 28 heads of 128, 2728 us with one announcement,
// 2504 us so. Announcing the first half before the third quarter's exponentials
// waits for the stores to TMEM with nothing to do: 2572 us; forming the first
// quarter with the old max while the new one is found: 2567 us.
template <int D>
__device__ __forceinline__ bool softmax_tile(const PrefillTcArgs& a, const Mask& mask,
                                             uint32_t tl, uint32_t s_col, uint32_t o_col, bool first, float& m,
                                             float& l, uint64_t* pv_done, uint32_t pv_parity,
                                             uint64_t* p_full, volatile int* abort_flag) {
  float s[kBN];
  {
    uint32_t v0[32], v1[32], v2[32], v3[32];
    tmem_ld32(tl + s_col, v0);
    tmem_ld32(tl + s_col + 32, v1);
    tmem_ld32(tl + s_col + 64, v2);
    tmem_ld32(tl + s_col + 96, v3);
    tmem_ld_wait();
#pragma unroll
    for (int e = 0; e < 32; ++e) {
      s[e] = __uint_as_float(v0[e]);
      s[32 + e] = __uint_as_float(v1[e]);
      s[64 + e] = __uint_as_float(v2[e]);
      s[96 + e] = __uint_as_float(v3[e]);
    }
  }
  tc_fence_before();

  // hidden keys -> -inf: four 32-bit masks (one per 32 keys), so that each score
  // costs one AND with an immediate and one select
  if (mask.need) {
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const uint32_t vm = range_bits(0, mask.e_hi - 32 * c) | range_bits(mask.a0 - 32 * c, mask.a1 - 32 * c) |
                          range_bits(mask.b0 - 32 * c, mask.b1 - 32 * c);
#pragma unroll
      for (int e = 0; e < 32; ++e) s[32 * c + e] = (vm & (1u << e)) ? s[32 * c + e] : -INFINITY;
    }
  }
  // p = 2^(s * scale - m), hidden keys give 0. Packed f32x2 arithmetic: one
  // FFMA2 forms two exponent arguments and one FADD2 adds two weights into
  // one of four pair accumulators. bf16 pairs (key k in column k/2, even k
  // low) are written over the first 64 columns of this tile's S in TMEM.
  const float2 sc2 = make_float2(a.scale_log2, a.scale_log2);
  float2 nm2, sum4[4];
  uint32_t w[16];
  auto form = [&](int hh) {
#pragma unroll
    for (int t = 0; t < 16; ++t) {
      const int k = hh * 32 + 2 * t;
      const float2 e = __ffma2_rn(make_float2(s[k], s[k + 1]), sc2, nm2);
      const float2 pp = make_float2(fast_exp2(e.x), fast_exp2(e.y));
      sum4[t & 3] = __fadd2_rn(sum4[t & 3], pp);
      w[t] = float2_to_bf16x2(pp.x, pp.y);
    }
  };
  // row max of the raw scores (the scale is positive): 8 chains of
  // three-input max
  float mx8[8];
#pragma unroll
  for (int u = 0; u < 8; ++u) mx8[u] = fmaxf(s[u], s[u + 8]);
#pragma unroll
  for (int k = 16; k < kBN; k += 16)
#pragma unroll
    for (int u = 0; u < 8; ++u) mx8[u] = fmax3f(mx8[u], s[k + u], s[k + 8 + u]);
  const float rmax = fmax3f(fmax3f(mx8[0], mx8[1], mx8[2]), fmax3f(mx8[3], mx8[4], mx8[5]), fmaxf(mx8[6], mx8[7])) *
                     a.scale_log2;
  const float mn = fmaxf(m, rmax);
  const bool resc = mn > m + kRescaleThreshold;
  float alpha = 1.f;
  if (__any_sync(0xffffffffu, resc)) {
    if (resc) {
      alpha = (m == -INFINITY) ? 0.f : fast_exp2(m - mn);
      m = mn;
    }
    // rescale O: the last O_X += P_X V must have landed first
    if (!first) {
      if (!__all_sync(0xffffffffu, wait_bar(pv_done, pv_parity, a.err, abort_flag))) return false;
      tc_fence_after();
#pragma unroll 1
      for (int c = 0; c < D / 8; ++c) {
        uint32_t v[8];
        tmem_ld8(tl + o_col + c * 8, v);
        tmem_ld_wait();
#pragma unroll
        for (int e = 0; e < 8; ++e) v[e] = __float_as_uint(__uint_as_float(v[e]) * alpha);
        tmem_st8(tl + o_col + c * 8, v);
      }
    }
  }
  const float neg_m = (m == -INFINITY) ? 0.f : -m;
  nm2 = make_float2(neg_m, neg_m);
#pragma unroll
  for (int u = 0; u < 4; ++u) sum4[u] = make_float2(0.f, 0.f);
  form(0);
  auto publish = [&](int half) {
    tmem_st_wait();
    tc_fence_before();
    __syncwarp();
    if ((threadIdx.x & 31) == 0) mbar_arrive(&p_full[half]);
  };
  tmem_st16(tl + s_col, w);
  form(1);
  tmem_st16(tl + s_col + 16, w);
  form(2);
  publish(0);  // keys 0-63, a third quarter's exponentials behind their stores
  tmem_st16(tl + s_col + 32, w);
  form(3);
  tmem_st16(tl + s_col + 48, w);
  publish(1);
  const float2 s01 = __fadd2_rn(sum4[0], sum4[1]), s23 = __fadd2_rn(sum4[2], sum4[3]);
  const float2 s03 = __fadd2_rn(s01, s23);
  const float sum = s03.x + s03.y;
  l = l * alpha + sum;

  return true;
}

// Output rows through shared memory: a warp's 32 rows of O come one to a lane,
// and lanes that each write their own row send 32 half-used sectors with every
// store (4,400 clocks at the end of an item, as much as 1.5 pairs of KV tiles).
// put_row stores 8 values of the lane's row as one of its 16-byte chunks, swizzled
// against bank conflicts; write_rows then stores whole rows, 256 bytes by 16
// lanes. 8 ragged sequences of up to 2,999 tokens: 313 -> 298 us; 32K tokens with
// streaming heads alone (S = 128, W = 1024) 570 -> 517 us.
template <int D>
__device__ __forceinline__ void put_row(uint8_t* stage, int lane, int chunk, const float (&y)[8]) {
  constexpr int CH = D / 8;
  uint4 w;
  w.x = float2_to_bf16x2(y[0], y[1]);
  w.y = float2_to_bf16x2(y[2], y[3]);
  w.z = float2_to_bf16x2(y[4], y[5]);
  w.w = float2_to_bf16x2(y[6], y[7]);
  *reinterpret_cast<uint4*>(stage + lane * (D * 2) + ((chunk ^ (lane % CH)) << 4)) = w;
}

// COLS columns, from col0 on, of rows i0 .. i0 + 31 of the chunk (those below len), query
// tile x's head, from the warp's `stage`.
template <int D, int COLS>
__device__ __forceinline__ void write_rows(const PrefillTcArgs& a, const Item& t, int x, int i0, int col0,
                                           const uint8_t* stage, int lane) {
  constexpr int CH = COLS / 8, RPI = 32 / CH;  // chunks a row, rows a step
  __syncwarp();
  const int c = lane % CH;
  bf16* out = static_cast<bf16*>(a.out) + ((size_t)t.b * a.T * a.geom.Hq + t.head(x)) * D + col0 + c * 8;
#pragma unroll
  for (int r0 = 0; r0 < 32; r0 += RPI) {
    const int r = r0 + lane / CH;
    const uint4 w = *reinterpret_cast<const uint4*>(stage + r * (COLS * 2) + ((c ^ (r % CH)) << 4));
    if (i0 + r < t.len) *reinterpret_cast<uint4*>(out + (size_t)(i0 + r) * a.geom.Hq * D) = w;
  }
}

// Write a warp's 32 finished rows of query tile x's O (each lane's times its inv), the
// first of them row i0 of the chunk, COLS columns at a time. taddr: O's first
// column, stage: 32 * COLS * 2 bytes.
template <int D, int COLS>
__device__ __forceinline__ void store_o(const PrefillTcArgs& a, const Item& t, int x, int i0, uint32_t taddr, float inv,
                                        uint8_t* stage, int lane) {
#pragma unroll
  for (int c = 0; c < D / 32; ++c) {
    uint32_t v[32];
    tmem_ld32(taddr + c * 32, v);
    tmem_ld_wait();
#pragma unroll
    for (int e = 0; e < 32; e += 8) {
      float y[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) y[k] = __uint_as_float(v[e + k]) * inv;
      put_row<COLS>(stage, lane, c % (COLS / 32) * 4 + e / 8, y);
    }
    if ((c + 1) * 32 % COLS == 0) {
      write_rows<D, COLS>(a, t, x, i0, (c + 1) * 32 - COLS, stage, lane);
      __syncwarp();
    }
  }
}

}  // namespace pf
}  // namespace aoh
