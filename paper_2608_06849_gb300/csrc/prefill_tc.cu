// Causal prefill attention on tcgen05 tensor cores (Sec. 5, "Chunked-Prefill
// Stage", with the per-token sink + window rule for streaming heads). A call
// processes one chunk of every sequence: rows at positions Lb .. Lb + len - 1
// after Lb cached tokens (Lb = 0 for a first prefill). Cached keys are read
// from the KV cache itself (retrieval rows, or the streaming sink + ring
// slots) before the chunk's own keys; the cache is appended after this
// kernel, so the ring still holds the positions the chunk's rows need.
//
// One CTA computes two 128-row query tiles (A, B) against the same stream of
// 128-key K/V tiles: the same rows of two heads of a group, or two consecutive
// tiles of one head. The KV tiles visited come from a per-head schedule: a
// retrieval head visits tiles 0 .. causal end; a streaming head only the
// tiles holding its S sinks and the tiles that intersect the W-token window
// of some row, so its cost is O(S + W) per row instead of O(T). Consecutive
// tiles visit the union of their tile sets; a tile hidden from every row of
// one query tile contributes zero weights there. Tiles fully visible to every
// row of a query tile skip the mask.
//
// Warp roles (320 threads):
//   warp 0      TMA producer: Q_A, Q_B once, then K_j / V_j tiles into a
//               4-stage ring (4D tensor maps over [B][T][H][D], 128-byte swizzle).
//   warp 1      TMEM owner and MMA issuer. S_X(j) = Q_X K_j^T reads both
//               operands from shared memory; O_X += P_X(j) V_j reads P_X from
//               TMEM, where the softmax wrote it over the first 64 columns of
//               S_X. Per KV tile the issue order is O_A += P_A V, S_A(j+1),
//               O_B += P_B V, S_B(j+1): a tile's next S overwrites its P only
//               after the P.V that reads it (MMAs of one thread run in order),
//               and while one query tile's softmax runs the tensor pipe works
//               on the other's MMAs, hiding the commit -> softmax -> issue
//               latency of each tile.
//   warps 2-5   softmax of tile A, warps 6-9 softmax of tile B: thread r owns
//               row r (TMEM lane r). One tcgen05.ld pass reads its S row, a
//               two-range integer mask hides keys, max and sum reduce in 8
//               independent chains, p = 2^(s*scale - m) costs one FFMA and one
//               EX2, the running max moves only when it grows by more than
//               2^8 (O rarely rescaled), and bf16 P pairs go back to TMEM with
//               tcgen05.st (key k in column k/2, even k in the low half),
//               announced in two halves of 64 keys.
// TMEM columns: S_A / P_A [0,128), S_B / P_B [128,256), O_A [256, 256+D),
// O_B [256+D, 256+2D).
#include <string.h>

#include "cluster.cuh"
#include "prefill_tile.cuh"

namespace aoh {
namespace {

using namespace pf;

// PAIRS: clusters of two CTAs, each with its entry of the list. Where both have the
// same item's halves, each visits half of its KV tiles; then each finishes one of
// the two query tiles: it receives the other
// CTA's state of that tile (O, running max and sum) in shared memory that the
// main loop no longer needs, adds its own and writes the rows.
template <int D, bool PAIRS, int CAP>
__global__ void __launch_bounds__(kThreads, 1)
    prefill_tc_kernel(const __grid_constant__ PrefillTcArgs a, const __grid_constant__ WorkList<CAP> wl) {
  using C = PfCfg<D>;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = smem_raw + ((1024 - (smem_u32(smem_raw) & 1023)) & 1023);
  uint8_t* sQ = smem + C::OFF_Q;
  uint8_t* sKV = smem + C::OFF_KV;
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + C::OFF_BAR);
  uint64_t* q_full = bars;
  uint64_t* kv_full = bars + 1;
  uint64_t* kv_empty = kv_full + kNS;
  uint64_t* s_full = kv_empty + kNS;  // [2]: S_A, S_B ready
  uint64_t* p_full = s_full + 2;      // [2][2]: P_A, P_B written, keys 0-63 and 64-127
  uint64_t* pv_done = p_full + 4;     // [2]: O_A, O_B updated (P buffer free)
  uint64_t* drain = pv_done + 2;
  // [2]: padding rows of the item's first / second partial V tile are zeroed.
  // Only the last cache tile and the chunk tile holding row len - 1 can be
  // partial, so each barrier completes at most once per item.
  uint64_t* v_zeroed = drain + 1;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(v_zeroed + 2);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // the append may start once the last CTAs of this grid run (append.cu)
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const uint64_t code = CAP > 0 ? wl.item[blockIdx.x] : a.work[blockIdx.x];
  if (PAIRS && code == kPrefillNone) return;
  const bool half = PAIRS && code >= kPrefillHalf;  // alike in both CTAs of a cluster
  const Item t(a, code & ~kPrefillHalf);
  const CacheGeom& g = a.geom;
  const int n_all = t.tiles();
  // this CTA visits tiles t0 .. t0 + n_tiles - 1 of the item's n_all
  const int rank = half ? (int)cluster_rank() : 0;
  const int t0 = rank * ((n_all + 1) / 2);
  const int n_tiles = !half ? n_all : rank == 0 ? (n_all + 1) / 2 : n_all / 2;
  if (threadIdx.x == 0) {
    mbar_init(q_full, 2);
    for (int s = 0; s < kNS; ++s) {
      mbar_init(&kv_full[s], 1);
      mbar_init(&kv_empty[s], 1);
    }
    for (int x = 0; x < 2; ++x) {
      mbar_init(&s_full[x], 1);
      mbar_init(&p_full[2 * x], 4);
      mbar_init(&p_full[2 * x + 1], 4);
      mbar_init(&pv_done[x], 1);
    }
    mbar_init(drain, 1);
    mbar_init(&v_zeroed[0], 1);
    mbar_init(&v_zeroed[1], 1);
    *abort_flag = 0;
    fence_mbar_init();
    fence_proxy_async_smem();
    // the first loads need no other warp
    load_q<D>(a, t, 0, sQ, q_full);
    load_q<D>(a, t, 1, sQ + C::QBYTES, q_full);
    if (n_tiles > 0) load_kv<D>(a, t, t0, 0, sKV, &kv_full[0]);
  }
  if (warp == 1) {
    tmem_alloc(tmem_slot, kTmemCols);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  // a half: a row's final softmax state (softmax warps)
  float end_m = -INFINITY, end_l = 0.f;
  bool end_ok = true;
  if (warp == 0) {
    // ------------------------------------------------------------ producer
    // Lane 0 issues the copies. Rows of a V tile past its valid keys may hold
    // anything (cache rows not yet written, chunk padding) and a zero weight
    // times a NaN is still NaN, so for a partial V tile the whole warp waits
    // for the copy, zeroes those rows and signals v_zeroed before the MMA
    // issuer may read the tile.
    int issued = min(n_tiles, 1), n_partial = 0;  // the first K tile is on its way
    bool ok = true;
    for (int jj = 0; jj < n_tiles && ok; ++jj) {
      for (int sel = 0; sel < 2; ++sel) {
        const int it = 2 * jj + sel;
        const int st = it % kNS;
        if (lane == 0) {
          if (it >= kNS) ok = wait_bar(&kv_empty[st], ((it / kNS) & 1) ^ 1, a.err, abort_flag);
          if (ok && it > 0) {
            load_kv<D>(a, t, t0 + jj, sel, sKV + st * C::KVBYTES, &kv_full[st]);
            issued = it + 1;
          }
        }
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
        const int valid = t.valid(g, t0 + jj);
        if (sel == 1 && valid < kBN && n_partial < 2) {
          ok = __all_sync(0xffffffffu, wait_bar(&kv_full[st], (it / kNS) & 1, a.err, abort_flag));
          if (!ok) break;
          zero_tail<D>(sKV + st * C::KVBYTES, valid, lane);
          if (lane == 0) mbar_arrive(&v_zeroed[n_partial]);
          ++n_partial;
        }
      }
    }
    // every issued copy lands before the CTA can exit
    if (lane == 0) {
      drain_wait(q_full, 0, a.err);
      for (int it = issued > kNS ? issued - kNS : 0; it < issued; ++it)
        drain_wait(&kv_full[it % kNS], (it / kNS) & 1, a.err);
    }
    __syncwarp();
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMA issuer
    // The whole warp runs the loop (its values stay warp-uniform); one elected
    // lane, the same each time, issues.
    const uint64_t q_desc = sdesc_sw128(smem_u32(sQ), 16, 1024);
    const uint64_t k_desc0 = sdesc_sw128(smem_u32(sKV), 16, 1024);
    const uint64_t v_desc0 = sdesc_sw128(smem_u32(sKV), C::BOX, 1024);
    auto s_of = [&](int x, int jj) {
      const uint64_t k_desc = k_desc0 + (uint32_t)(((2 * jj) % kNS) * sdesc_step(C::KVBYTES));
      if (elect_one()) {
        issue_s<D>(tmem, q_desc + sdesc_step(x * C::QBYTES), k_desc, x);
        tc_commit(&s_full[x]);
      }
    };
    auto commit = [&](uint64_t* bar) {
      if (elect_one()) tc_commit(bar);
    };
    bool ok = n_tiles > 0;
    auto wait = [&](uint64_t* bar, uint32_t parity) {
      if (ok) ok = __all_sync(0xffffffffu, wait_bar(bar, parity, a.err, abort_flag));
      return ok;
    };
    // O_X += P_X(jj) V_jj: the first half of the keys while the softmax forms the
    // second half's weights
    auto pv_of = [&](int x, int jj) {
      const uint64_t v_desc = v_desc0 + (uint32_t)(((2 * jj + 1) % kNS) * sdesc_step(C::KVBYTES));
#pragma unroll
      for (int half = 0; half < 2; ++half) {
        if (!wait(&p_full[2 * x + half], jj & 1)) return false;
        tc_fence_after();
        if (elect_one()) {
          issue_pv<D>(tmem, v_desc, x, half, jj == 0);
          if (half) tc_commit(&pv_done[x]);
        }
      }
      return true;
    };
    auto wait_k = [&](int jj) { return wait(&kv_full[(2 * jj) % kNS], ((2 * jj) / kNS) & 1); };
    // only the last cached tile and the last chunk tile can be partial
    int n_partial = 0;  // partial V tiles seen so far (index into v_zeroed)
    const int part0 = t.n_c > 0 && t.valid(g, t.n_c - 1) < kBN ? t.n_c - 1 - t0 : -1;
    const int part1 = t.valid(g, n_all - 1) < kBN ? n_all - 1 - t0 : -1;
    auto wait_v = [&](int jj) {
      if (!wait(&kv_full[(2 * jj + 1) % kNS], ((2 * jj + 1) / kNS) & 1)) return false;
      if (jj == part0 || jj == part1) {
        if (!wait(&v_zeroed[n_partial], 0)) return false;
        ++n_partial;
      }
      return true;
    };
    if (wait(q_full, 0) && wait_k(0)) {
      tc_fence_after();
      s_of(0, 0);
      s_of(1, 0);
      commit(&kv_empty[0]);
    }
    for (int jj = 0; jj < n_tiles && ok; ++jj) {
      const bool more = jj + 1 < n_tiles;
      // tile A: P_A(jj) sits in S_A's columns; S_A(jj+1) may overwrite them
      // only after O_A += P_A(jj) V_jj is issued (same-thread MMAs run in order)
      if (!wait_v(jj) || !pv_of(0, jj)) break;
      if (more) {
        if (!wait_k(jj + 1)) break;
        tc_fence_after();
        s_of(0, jj + 1);
      }
      if (!pv_of(1, jj)) break;
      commit(&kv_empty[(2 * jj + 1) % kNS]);
      if (more) {
        s_of(1, jj + 1);
        commit(&kv_empty[(2 * (jj + 1)) % kNS]);
      }
    }
    commit(drain);
    __syncwarp();
    drain_wait(drain, 0, a.err);
    __syncwarp();
  } else {
    // ------------------------------------------------------------ softmax
    const int x = (warp - 2) >> 2;        // 0: tile A (warps 2-5), 1: tile B (warps 6-9)
    const int q4 = warp & 3;              // TMEM lane quarter this warp may access
    const int r = q4 * 32 + lane;
    const int qx0 = t.row0(x);            // first row of this query tile
    const int i = qx0 + r;
    const uint32_t tl = tmem + ((uint32_t)(q4 * 32) << 16);
    const uint32_t s_col = x * 128, o_col = 256 + x * D;
    const int rot = (t.streaming && t.Lb > g.S + g.W) ? (t.Lb - g.S) % g.W : 0;
    float m = -INFINITY, l = 0.f;
    bool ok = true;
    for (int jj = 0; jj < n_tiles && ok; ++jj) {
      const Mask mask(g, t, t0 + jj, i, qx0, rot);
      ok = __all_sync(0xffffffffu, wait_bar(&s_full[x], jj & 1, a.err, abort_flag));
      if (!ok) break;
      tc_fence_after();
      ok = softmax_tile<D>(a, mask, tl, s_col, o_col, jj == 0, m, l, &pv_done[x], (jj - 1) & 1,
                           &p_full[2 * x], abort_flag);
    }
    if (half) {
      end_m = m;
      end_l = l;
      end_ok = ok && (n_tiles == 0 ||
                      __all_sync(0xffffffffu, wait_bar(&pv_done[x], (n_tiles - 1) & 1, a.err, abort_flag)));
    } else if (ok && __all_sync(0xffffffffu, wait_bar(&pv_done[x], (n_tiles - 1) & 1, a.err, abort_flag))) {
      tc_fence_after();
      // Q_X is free: the last S_X was done before the last P V
      store_o<D, D>(a, t, x, qx0 + q4 * 32, tl + o_col, 1.f / l, sQ + x * C::QBYTES + q4 * (C::QBYTES / 4), lane);
    }
  }

  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (half) {
    // both CTAs' copies and MMAs are done with their shared memory
    cluster_arrive();
    cluster_wait();
    const int x = (warp - 2) >> 2, q4 = warp & 3, r = q4 * 32 + lane;
    const uint32_t tl = tmem + ((uint32_t)(q4 * 32) << 16) + 256 + x * D;
    float4* recv = reinterpret_cast<float4*>(smem);  // [D / 4][128 rows], then (m, l) per row
    float2* recv_ml = reinterpret_cast<float2*>(recv + D / 4 * 128);
    if (warp >= 2 && x != rank) {
      const uint32_t dst = cluster_addr(recv + r, (uint32_t)(rank ^ 1));
      cluster_st2(cluster_addr(recv_ml + r, (uint32_t)(rank ^ 1)), __float_as_uint(end_m), __float_as_uint(end_l));
      if (n_tiles > 0) {
#pragma unroll
        for (int c = 0; c < D / 32; ++c) {
          uint32_t v[32];
          tmem_ld32(tl + c * 32, v);
          tmem_ld_wait();
#pragma unroll
          for (int e = 0; e < 32; e += 4)
            cluster_st4(dst + (uint32_t)((c * 8 + e / 4) * 128 * 16), v[e], v[e + 1], v[e + 2], v[e + 3]);
        }
      }
      tc_fence_before();
    }
    cluster_arrive();
    cluster_wait();
    if (warp >= 2 && x == rank && end_ok) {
      const float2 o_ml = recv_ml[r];
      const float M = fmaxf(end_m, o_ml.x);
      // a state of -inf saw no key of this row, and its CTA may have had no tile at all
      // (unwritten values); any other state counts, also with a weight that rounds to
      // zero, whose NaN is one in a single CTA as well
      const bool mine = end_m != -INFINITY, other = o_ml.x != -INFINITY;
      const float w0 = mine ? fast_exp2(end_m - M) : 0.f, w1 = other ? fast_exp2(o_ml.x - M) : 0.f;
      const float inv = 1.f / (end_l * w0 + o_ml.y * w1);
      const float f0 = w0 * inv, f1 = w1 * inv;
      uint8_t* stage = smem + C::OFF_BAR - C::QBYTES + q4 * (C::QBYTES / 4);  // past the receive buffer
#pragma unroll
      for (int c = 0; c < D / 32; ++c) {
        uint32_t v[32];
        tmem_ld32(tl + c * 32, v);
        tmem_ld_wait();
#pragma unroll
        for (int e = 0; e < 32; e += 8) {
          float y[8];
#pragma unroll
          for (int k = 0; k < 8; k += 4) {
            const float4 z = recv[(c * 8 + (e + k) / 4) * 128 + r];
            y[k + 0] = (mine ? __uint_as_float(v[e + k + 0]) * f0 : 0.f) + (other ? z.x * f1 : 0.f);
            y[k + 1] = (mine ? __uint_as_float(v[e + k + 1]) * f0 : 0.f) + (other ? z.y * f1 : 0.f);
            y[k + 2] = (mine ? __uint_as_float(v[e + k + 2]) * f0 : 0.f) + (other ? z.z * f1 : 0.f);
            y[k + 3] = (mine ? __uint_as_float(v[e + k + 3]) * f0 : 0.f) + (other ? z.w * f1 : 0.f);
          }
          put_row<D>(stage, lane, c * 4 + e / 8, y);
        }
      }
      write_rows<D, D>(a, t, x, t.row0(x) + q4 * 32, 0, stage, lane);
      tc_fence_before();
    }
    __syncthreads();
    tc_fence_after();
  }
  if (warp == 1) tmem_dealloc(tmem, kTmemCols);
}

}  // namespace

PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  if (!fn) {
    cudaDriverEntryPointQueryResult q;
    void* p = nullptr;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
            cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
  }
  return fn;
}

namespace {

// 4D map over a [B][T][H][D] bf16 tensor, box [1][128][1][64], 128-byte swizzle.
bool make_map(CUtensorMap* map, const void* base, int B, int T, int H, int D) {
  auto fn = encode_fn();
  if (!fn) return false;
  cuuint64_t dims[4] = {(cuuint64_t)D, (cuuint64_t)H, (cuuint64_t)T, (cuuint64_t)B};
  cuuint64_t strides[3] = {(cuuint64_t)D * 2, (cuuint64_t)H * D * 2, (cuuint64_t)T * H * D * 2};
  cuuint32_t box[4] = {64, 1, 128, 1};
  cuuint32_t estr[4] = {1, 1, 1, 1};
  CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(base), dims, strides, box, estr,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}

constexpr int kSmall = 640;  // items of a launch that copies 5 KB of arguments instead of 30

template <int D, bool PAIRS, int CAP>
cudaError_t launch_cfg(const PrefillTcArgs& a, const std::vector<uint64_t>& items, cudaStream_t s) {
  using C = PfCfg<D>;
  static std::atomic<uint64_t> done{0};
  const cudaError_t e = once_per_device(done, [] {
    return cudaFuncSetAttribute(prefill_tc_kernel<D, PAIRS, CAP>, cudaFuncAttributeMaxDynamicSharedMemorySize, C::SMEM);
  });
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)items.size());
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = C::SMEM;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2;
  attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = PAIRS ? 1 : 0;
  WorkList<CAP> wl;
  if (CAP > 0) memcpy(wl.item, items.data(), items.size() * sizeof(uint64_t));
  return cudaLaunchKernelEx(&cfg, prefill_tc_kernel<D, PAIRS, CAP>, a, wl);
}

template <int D>
cudaError_t launch_d(const PrefillTcArgs& a, const std::vector<uint64_t>& items, const std::vector<uint64_t>& pairs,
                     cudaStream_t s) {
  if (!pairs.empty()) return launch_cfg<D, true, 2 * kPrefillSplitMost>(a, pairs, s);
  if (items.size() <= kSmall) return launch_cfg<D, false, kSmall>(a, items, s);
  if (items.size() <= kPrefillByValue) return launch_cfg<D, false, kPrefillByValue>(a, items, s);
  return launch_cfg<D, false, 0>(a, items, s);
}

}  // namespace

bool prefill_tc_make_maps(PrefillTcArgs* a, const void* q, const void* k, const void* v, int B, int T) {
  const CacheGeom& g = a->geom;
  return make_map(&a->tq, q, B, T, g.Hq, g.D) && make_map(&a->tk, k, B, T, g.Hkv, g.D) &&
         make_map(&a->tv, v, B, T, g.Hkv, g.D);
}

// 4D map over one kind of cache region: [regions][K, V][cap rows][D], box
// [1][1][128][64], 128-byte swizzle. Rows past `cap` read as zeros.
// With `step` 2 the map holds every second of the cap rows, `base` being the
// first of them and `rows` their number.
static bool make_region_map(CUtensorMap* map, const void* base, int regions, int cap, int D, int step = 1,
                            int rows = 0) {
  auto fn = encode_fn();
  if (!fn) return false;
  if (step == 1) rows = cap;
  cuuint64_t dims[4] = {(cuuint64_t)D, (cuuint64_t)rows, 2, (cuuint64_t)regions};
  cuuint64_t strides[3] = {(cuuint64_t)D * 2 * step, (cuuint64_t)cap * D * 2, (cuuint64_t)cap * D * 2 * 2};
  cuuint32_t box[4] = {64, 128, 1, 1};
  cuuint32_t estr[4] = {1, 1, 1, 1};
  CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(base), dims, strides, box, estr,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}

bool make_cache_region_maps(CUtensorMap* tcr, CUtensorMap* tcs, const CacheGeom& g, const void* kv) {
  const bf16* base = static_cast<const bf16*>(kv);
  bool ok = true;
  if (g.n_r > 0) ok = ok && make_region_map(tcr, base + g.r_region(0, 0), g.B * g.n_r, g.max_seq, g.D);
  if (g.n_s > 0) ok = ok && make_region_map(tcs, base + g.s_region(0, 0), g.B * g.n_s, g.S + g.W, g.D);
  return ok;
}

bool make_decode_maps(DecodeArgs* a, const CacheGeom& g, const void* kv) {
  if (g.D != 64) return make_cache_region_maps(&a->tcr, &a->tcs, g, kv);
  const bf16* base = static_cast<const bf16*>(kv);
  bool ok = true;
  for (int odd = 0; odd < 2; ++odd) {
    auto pair_map = [&](CUtensorMap* map, const bf16* first, int regions, int cap) {
      // a region of one row has no odd row: its map repeats the even one
      const int shift = odd && cap > 1 ? g.D : 0;
      return make_region_map(map, first + shift, regions, cap, g.D, 2, odd && cap > 1 ? cap / 2 : (cap + 1) / 2);
    };
    if (g.n_r > 0)
      ok = ok && pair_map(odd ? &a->tcr_odd : &a->tcr, base + g.r_region(0, 0), g.B * g.n_r, g.max_seq);
    if (g.n_s > 0)
      ok = ok && pair_map(odd ? &a->tcs_odd : &a->tcs, base + g.s_region(0, 0), g.B * g.n_s, g.S + g.W);
  }
  return ok;
}

bool prefill_tc_make_cache_maps(PrefillTcArgs* a, const void* kv) {
  return make_cache_region_maps(&a->tcr, &a->tcs, a->geom, kv);
}

cudaError_t launch_prefill_tc(const PrefillTcArgs& a, const std::vector<uint64_t>& items,
                              const std::vector<uint64_t>& pairs, cudaStream_t s) {
  if (items.empty()) return cudaSuccess;
  if (a.geom.D == 128) return launch_d<128>(a, items, pairs, s);
  if (a.geom.D == 64) return launch_d<64>(a, items, pairs, s);
  return cudaErrorInvalidValue;
}

}  // namespace aoh
