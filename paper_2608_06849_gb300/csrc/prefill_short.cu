// Prefill of many short work items (prefill_tc.cu describes the computation and
// the warps' roles): one CTA an SM goes through its items in one pipeline. A CTA an
// item spends 4 us of its life on its start (barriers, TMEM, Q and the first tile
// from memory, the first S and its softmax) and its end (the last P V, O to
// memory) with idle tensor cores, as much as three KV tiles of work. Here the next
// item's K, V and Q load while the last tiles of this one run, and a query tile's
// rows are written while the other's MMAs and the next item's first S go on.
//
// Barrier phases run on across items (counters instead of tile indexes); q_empty
// tells the producer that the item's last S is done. O needs no barrier: the warps
// that read O_X are those whose weights the next item's first P V into it waits
// for. The items are dealt in a fixed order, heaviest first, forth and back (CTA c
// takes items c, 2 P - 1 - c, 2 P + c, ...), which evens out their cost.
//
// 8 ragged sequences of up to 2,999 tokens, 32/8 heads of 128 of which half stream (S =
// 64, W = 512): 276 us with a CTA an item, 244 so; heads of 64 230 -> 210; 16 sequences
// of up to 700 tokens 89 -> 71. What is left of an item's start and end is the chain
// from its last S to the next item's first P V: Q's buffer, S and its softmax.
#include <string.h>

#include "prefill_tile.cuh"

namespace aoh {
namespace {

using namespace pf;

template <int D>
struct ShortCfg {
  using C = PfCfg<D>;
  static constexpr int COLS = 64;                // columns of O staged at a time
  static constexpr int STAGE = 32 * COLS * 2;    // a warp's
  static constexpr int OFF_STAGE = C::OFF_BAR;   // 8 warps
  static constexpr int OFF_BAR = OFF_STAGE + 8 * STAGE;
  static constexpr int NBAR = 2 + 2 * kNS + 2 + 4 + 2 + 2 + 1;
  static constexpr int SMEM = OFF_BAR + NBAR * 8 + 16 + 1024;
  static_assert(SMEM <= 232448, "shared memory");
};

template <int D, int CAP>
__global__ void __launch_bounds__(kThreads, 1)
    prefill_short_kernel(const __grid_constant__ PrefillTcArgs a, const __grid_constant__ WorkList<CAP> wl, int n_items) {
  using C = PfCfg<D>;
  using X = ShortCfg<D>;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = smem_raw + ((1024 - (smem_u32(smem_raw) & 1023)) & 1023);
  uint8_t* sQ = smem + C::OFF_Q;
  uint8_t* sKV = smem + C::OFF_KV;
  uint64_t* q_full = reinterpret_cast<uint64_t*>(smem + X::OFF_BAR);
  uint64_t* q_empty = q_full + 1;
  uint64_t* kv_full = q_empty + 1;
  uint64_t* kv_empty = kv_full + kNS;
  uint64_t* s_full = kv_empty + kNS;   // [2]: S_A, S_B ready
  uint64_t* p_full = s_full + 2;       // [2][2]: P_A, P_B written, keys 0-63 and 64-127
  uint64_t* pv_done = p_full + 4;      // [2]: O_A, O_B updated
  uint64_t* v_zeroed = pv_done + 2;    // [2]: padding rows of every other partial V tile are zeroed
  uint64_t* drain = v_zeroed + 2;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(drain + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const CacheGeom& g = a.geom;
  const int P = gridDim.x, cta = blockIdx.x;
  // this CTA's k-th item
  auto item_index = [&](int k) { return k * P + ((k & 1) ? P - 1 - cta : cta); };
  auto item_code = [&](int i) { return CAP > 0 ? wl.item[i] : a.work[i]; };
  if (threadIdx.x == 0) {
    mbar_init(q_full, 2);
    mbar_init(q_empty, 1);
    for (int s = 0; s < kNS; ++s) {
      mbar_init(&kv_full[s], 1);
      mbar_init(&kv_empty[s], 1);
    }
    for (int x = 0; x < 2; ++x) {
      mbar_init(&s_full[x], 1);
      mbar_init(&p_full[2 * x], 4);
      mbar_init(&p_full[2 * x + 1], 4);
      mbar_init(&pv_done[x], 1);
      mbar_init(&v_zeroed[x], 1);
    }
    mbar_init(drain, 1);
    *abort_flag = 0;
    fence_mbar_init();
  }
  if (warp == 1) {
    tmem_alloc(tmem_slot, kTmemCols);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  if (warp == 0) {
    // ------------------------------------------------------------ producer
    int it = 0;         // copies of the KV ring so far (K, V, K, V, ...)
    int n_partial = 0;  // partial V tiles so far
    int issued = 0, nq = 0;
    bool ok = true;
    for (int k = 0; ok; ++k) {
      const int ii = item_index(k);
      if (ii >= n_items) break;
      // the append may start once every CTA is at its last item (append.cu)
      if (item_index(k + 1) >= n_items) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
      const Item t(a, item_code(ii));
      const int n = t.tiles();
      for (int jj = 0; jj < n && ok; ++jj) {
        for (int sel = 0; sel < 2; ++sel, ++it) {
          const int st = it % kNS;
          if (lane == 0) {
            if (it >= kNS) ok = wait_bar(&kv_empty[st], ((it / kNS) & 1) ^ 1, a.err, abort_flag);
            if (ok) {
              load_kv<D>(a, t, jj, sel, sKV + st * C::KVBYTES, &kv_full[st]);
              issued = it + 1;
            }
            if (ok && jj == 0 && sel == 0) {
              // Q after the first K tile: its buffer is free once the last
              // item's last S is done
              if (k >= 1) ok = wait_bar(q_empty, (k - 1) & 1, a.err, abort_flag);
              if (ok) {
                load_q<D>(a, t, 0, sQ, q_full);
                load_q<D>(a, t, 1, sQ + C::QBYTES, q_full);
                nq = k + 1;
              }
            }
          }
          ok = __all_sync(0xffffffffu, ok);
          if (!ok) break;
          const int valid = t.valid(g, jj);
          if (sel == 1 && valid < kBN) {
            ok = __all_sync(0xffffffffu, wait_bar(&kv_full[st], (it / kNS) & 1, a.err, abort_flag));
            if (!ok) break;
            zero_tail<D>(sKV + st * C::KVBYTES, valid, lane);
            if (lane == 0) mbar_arrive(&v_zeroed[n_partial & 1]);
            ++n_partial;
          }
        }
      }
    }
    // every issued copy lands before the CTA can exit
    if (lane == 0) {
      if (nq > 0) drain_wait(q_full, (nq - 1) & 1, a.err);
      for (int j = issued > kNS ? issued - kNS : 0; j < issued; ++j)
        drain_wait(&kv_full[j % kNS], (j / kNS) & 1, a.err);
    }
    __syncwarp();
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMA issuer
    const uint64_t q_desc = sdesc_sw128(smem_u32(sQ), 16, 1024);
    const uint64_t k_desc0 = sdesc_sw128(smem_u32(sKV), 16, 1024);
    const uint64_t v_desc0 = sdesc_sw128(smem_u32(sKV), C::BOX, 1024);
    int kt = 0;         // KV tiles before this one, over all items
    int n_partial = 0;  // partial V tiles so far
    bool ok = true;
    auto wait = [&](uint64_t* bar, uint32_t parity) {
      if (ok) ok = __all_sync(0xffffffffu, wait_bar(bar, parity, a.err, abort_flag));
      return ok;
    };
    auto commit = [&](uint64_t* bar) {
      if (elect_one()) tc_commit(bar);
    };
    auto s_of = [&](int x, int kt) {
      const uint64_t k_desc = k_desc0 + (uint32_t)(((2 * kt) % kNS) * sdesc_step(C::KVBYTES));
      if (elect_one()) {
        issue_s<D>(tmem, q_desc + sdesc_step(x * C::QBYTES), k_desc, x);
        tc_commit(&s_full[x]);
      }
    };
    auto pv_of = [&](int x, bool first) {
      const uint64_t v_desc = v_desc0 + (uint32_t)(((2 * kt + 1) % kNS) * sdesc_step(C::KVBYTES));
#pragma unroll
      for (int half = 0; half < 2; ++half) {
        if (!wait(&p_full[2 * x + half], kt & 1)) return false;
        tc_fence_after();
        if (elect_one()) {
          issue_pv<D>(tmem, v_desc, x, half, first);
          if (half) tc_commit(&pv_done[x]);
        }
      }
      return true;
    };
    auto wait_k = [&](int kt) { return wait(&kv_full[(2 * kt) % kNS], ((2 * kt) / kNS) & 1); };
    for (int k = 0; ok; ++k) {
      const int ii = item_index(k);
      if (ii >= n_items) break;
      const Item t(a, item_code(ii));
      const int n = t.tiles();
      const int part0 = t.n_c > 0 && t.valid(g, t.n_c - 1) < kBN ? t.n_c - 1 : -1;
      const int part1 = t.valid(g, n - 1) < kBN ? n - 1 : -1;
      if (!wait(q_full, k & 1) || !wait_k(kt)) break;
      tc_fence_after();
      s_of(0, kt);
      s_of(1, kt);
      commit(&kv_empty[(2 * kt) % kNS]);
      if (n == 1) commit(q_empty);
      for (int jj = 0; jj < n && ok; ++jj, ++kt) {
        const bool more = jj + 1 < n;
        if (!wait(&kv_full[(2 * kt + 1) % kNS], ((2 * kt + 1) / kNS) & 1)) break;
        if (jj == part0 || jj == part1) {
          if (!wait(&v_zeroed[n_partial & 1], (n_partial >> 1) & 1)) break;
          ++n_partial;
        }
        if (!pv_of(0, jj == 0)) break;
        if (more) {
          if (!wait_k(kt + 1)) break;
          tc_fence_after();
          s_of(0, kt + 1);
        }
        if (!pv_of(1, jj == 0)) break;
        commit(&kv_empty[(2 * kt + 1) % kNS]);
        if (more) {
          s_of(1, kt + 1);
          commit(&kv_empty[(2 * (kt + 1)) % kNS]);
          if (jj + 2 == n) commit(q_empty);
        }
      }
    }
    commit(drain);
    __syncwarp();
    drain_wait(drain, 0, a.err);
    __syncwarp();
  } else {
    // ------------------------------------------------------------ softmax
    const int x = (warp - 2) >> 2;  // 0: tile A (warps 2-5), 1: tile B (warps 6-9)
    const int q4 = warp & 3;        // TMEM lane quarter this warp may access
    const int r = q4 * 32 + lane;
    const uint32_t tl = tmem + ((uint32_t)(q4 * 32) << 16);
    const uint32_t s_col = x * 128, o_col = 256 + x * D;
    uint8_t* stage = smem + X::OFF_STAGE + (warp - 2) * X::STAGE;
    uint32_t kt = 0;  // KV tiles so far, over all items
    bool ok = true;
    for (int k = 0; ok; ++k) {
      const int ii = item_index(k);
      if (ii >= n_items) break;
      const Item t(a, item_code(ii));
      const int qx0 = t.row0(x), i = qx0 + r, n = t.tiles();
      const int rot = (t.streaming && t.Lb > g.S + g.W) ? (t.Lb - g.S) % g.W : 0;
      float m = -INFINITY, l = 0.f;
      for (int jj = 0; jj < n && ok; ++jj, ++kt) {
        const Mask mask(g, t, jj, i, qx0, rot);
        ok = __all_sync(0xffffffffu, wait_bar(&s_full[x], kt & 1, a.err, abort_flag));
        if (!ok) break;
        tc_fence_after();
        ok = softmax_tile<D>(a, mask, tl, s_col, o_col, jj == 0, m, l, &pv_done[x], (kt - 1) & 1, &p_full[2 * x],
                             abort_flag);
      }
      if (!ok) break;
      ok = __all_sync(0xffffffffu, wait_bar(&pv_done[x], (kt - 1) & 1, a.err, abort_flag));
      if (!ok) break;
      tc_fence_after();
      store_o<D, X::COLS>(a, t, x, qx0 + q4 * 32, tl + o_col, 1.f / l, stage, lane);
      tc_fence_before();
    }
  }

  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 1) tmem_dealloc(tmem, kTmemCols);
}

template <int D, int CAP>
cudaError_t launch_short_cfg(const PrefillTcArgs& a, const std::vector<uint64_t>& items, int num_sms, cudaStream_t s) {
  using X = ShortCfg<D>;
  static std::atomic<uint64_t> done{0};
  const cudaError_t e = once_per_device(done, [] {
    return cudaFuncSetAttribute(prefill_short_kernel<D, CAP>, cudaFuncAttributeMaxDynamicSharedMemorySize, X::SMEM);
  });
  if (e != cudaSuccess) return e;
  const int n = (int)items.size();
  WorkList<CAP> wl;
  if (CAP > 0) memcpy(wl.item, items.data(), items.size() * sizeof(uint64_t));
  prefill_short_kernel<D, CAP><<<n < num_sms ? n : num_sms, kThreads, X::SMEM, s>>>(a, wl, n);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_prefill_short(const PrefillTcArgs& a, const std::vector<uint64_t>& items, int num_sms,
                                 cudaStream_t s) {
  const bool by_value = items.size() <= (size_t)kPrefillByValue;
  if (a.geom.D == 128)
    return by_value ? launch_short_cfg<128, kPrefillByValue>(a, items, num_sms, s)
                    : launch_short_cfg<128, 0>(a, items, num_sms, s);
  if (a.geom.D == 64)
    return by_value ? launch_short_cfg<64, kPrefillByValue>(a, items, num_sms, s)
                    : launch_short_cfg<64, 0>(a, items, num_sms, s);
  return cudaErrorInvalidValue;
}

}  // namespace aoh
