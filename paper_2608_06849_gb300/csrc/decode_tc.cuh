// Split-KV decode on tcgen05 tensor cores (Sec. 5, "Decode Stage", Eq. 8;
// d_head 128 with GQA groups of 1-8 and 16, d_head 64 with 1, 2, 4, 7 and 8). With G query heads per KV head,
// every cached K/V row meets G queries: 4*G*d flops per 4*d bytes. On CUDA
// cores that arithmetic (plus the shuffles that reduce the dot products)
// stops hiding under the HBM stream above g = 4, and even at g = 4 it costs a
// few percent; here it runs as two skinny MMAs per 128-key tile, with the G
// heads padded to N = 16:
//
//   S^T[128 keys][16]  = K_tile[128][d] . Q^T           (A = K, K-major; B = Q, K-major)
//   O^T[d][16]        += V_tile^T[d][128] . P^T[128][16] (A = V, MN-major; B = P, K-major)
//
// (d_head 128; d_head 64 puts two keys into an MMA row, see Lay.)
// Both accumulators live in TMEM: S^T in one of two 16-column buffers (row =
// key), O^T in 16 more columns (row = d). The split of the step's rows over
// CTAs, the partial format and the merge are those of the CUDA-core kernel
// (decode_common.cuh); one CTA per SM.
//
// Warp roles (192 threads; 704 in the reuse step's variant for G <= 4, 448
// above):
//   warps 0-3  softmax: thread t owns key t of the tile (TMEM lane t). It
//              reads its 16 scores, hides keys past the tile's valid rows,
//              takes the per-head tile maximum (warp redux, then the four
//              warps through shared memory), moves the running maximum only
//              when it grows by more than 2^8 (then rescales its row d = t of
//              O^T in TMEM), forms p = 2^(s - m) and writes P^T as bf16 into a
//              swizzled K-major [16][128] buffer. Per-thread partial sums of p
//              are reduced once per item. Rows past the valid keys of a tail V
//              tile are zeroed first: they may hold unwritten cache rows and a
//              zero weight times a NaN is NaN.
//   warp 4     TMA producer: K and V tiles of one (sequence, KV head) region
//              into a 3-stage ring (4D tensor maps over the cache regions,
//              128-byte swizzle, rows past the region read as zeros).
//   warps 6-21 (6-13 for G > 4; the H2Share reuse step's variant) gather
//              warps: a retrieval item's rows are borrowed positions, which
//              these warps copy with 16-byte cp.async copies into the same
//              swizzled ring, 8 (16) rows of each tile per warp; the CTAs
//              split the step's rows with each gathered row weighing 3/2
//              contiguous rows (a row gather costs more than its share of a
//              streamed tile). The MMA warp issues a gathered tile's P V
//              right after its P, which frees the ring stage for the next
//              gather one tile earlier.
//   warp 5     TMEM owner and MMA issuer. Loads each item's Q into one of two
//              swizzled buffers, writes the new token's K/V row over its
//              (stale) cache row in the landed tile and appends it to the
//              cache, issues S(j) and then O += P(j-1) V(j-1).
#pragma once

#include <math.h>

#include "cluster.cuh"
#include "common.cuh"
#include "decode_common.cuh"
#include "internal.h"
#include "tc.cuh"

namespace aoh {
namespace dtc {

using bf16 = __nv_bfloat16;
constexpr int kBN = 128;                   // keys per tile
constexpr int kN = 16;                     // N of both MMAs (query heads, padded)
constexpr int kNS = 3;                     // ring stages
constexpr int kThreads = 192;              // warps 0-5 (see the file comment)
constexpr int kSoftmaxThreads = 128;
constexpr float kRescaleThreshold = 8.0f;  // log2 units
// Rows charged for a switch from one item to the next (DecodeArgs::
// item_cost), in steps whose CTAs hold fewer than kItemCostMaxShare rows
// each. A CTA that switches finishes its first item's epilogue and arrival
// before the next item's softmax can go on, so with an equal share it ends
// last, and then also runs the second item's merge. Measured with B=1,
// Qwen2.5-7B shape (2 of 4 KV heads streaming), us per step, mean over six
// lengths T .. T + 331 (cost 0 / 256 / 384 / 512 / 768 rows): 4K 16.9 /
// 16.9 / 16.2 / 15.4 / 14.9, 8K 23.2 / 20.5 / 17.8 / 17.0 / 15.7, 16K 19.9
// / 17.8 / 17.3 / 17.3 / 17.4, 32K 21.7 / 18.1 / 18.0 / 17.8 / 17.8, 64K
// 24.7 / 23.8 / 22.7 / 22.9 / 22.9, 128K 38.2 / - / 36.9 / 37.5 / 37.5;
// through the 28-layer stack per token (CUDA graph; cost 384 / 512 / 768):
// 4K 439 / 432 / 399, 32K 531 / 531 / 528, 128K 973 / 1037 / 1030.
// Steps on fewer CTAs than SMs (4K, 8K: at least 512 rows per CTA, few
// items) gain from the larger charge, which moves item starts onto CTA
// boundaries; steps on every SM keep 384. Llama-3-8B shape at B=16, 128K
// (29K rows per CTA): 628 us with no charge, 629-630 with 256 rows.
constexpr int kItemCost = 384;
constexpr int kItemCostFewCtas = 768;
constexpr long long kItemCostMaxShare = 16384;
constexpr int kBox = kBN * 64 * 2;         // one [128 rows][64] TMA box, 16 KB
constexpr int kTile = 2 * kBox;            // a K or V tile (d = 128)
constexpr int kStage = 2 * kTile;          // K then V

// Shapes and shared memory of one head size and group. At d_head 128 an MMA row
// is one key. At d_head 64 it is a pair of neighbouring keys, whose two 128-byte
// rows fill the two 64-wide column blocks of the same tile: the scores of the
// even and of the odd keys are two MMA sets over one block each, and P has a
// column per head and parity. O^T then holds the even keys' sum in rows 0-63 of
// the even columns and the odd keys' in rows 64-127 of the odd ones (the other
// halves are not used). P keeps its 24 bits at d_head 64: each weight is the
// sum of three bf16 parts, each a column of its own (outputs as close to 64 bits
// as with fp32 weights: both are the rounded exact value in 99.9% of 2,048
// outputs at 100K keys). On CUDA cores this head size was bound by the shuffles
// and FMAs of the dot products, 3.6 TB/s where this kernel reaches 5.0: a step
// of 8 sequences of 12K-32K keys, 32/8 heads, half of them streaming (213 MB),
// went from 59.5 to 45.7 us, a length copy included.
template <int D, int G>
struct Lay {
  static constexpr bool PAIR = D == 64;
  static constexpr int NK = PAIR ? 2 : 1;                      // keys per MMA row
  static constexpr int PARTS = PAIR ? 3 : 1;                   // bf16 parts of a weight
  static constexpr int HP = PAIR ? (G <= 4 ? 4 : 8) : kN;      // P columns of one parity
  static constexpr int NP = NK * HP;                           // P columns of one part
  static constexpr int NPV = (PARTS * NP + 15) / 16 * 16;      // N of the P V MMA
  static constexpr int SCOLS = NK * kN;                        // TMEM columns of an S buffer
  static constexpr uint32_t OCOL = 2 * SCOLS;                  // O after S[0], S[1]
  static constexpr uint32_t TMEM_COLS = PAIR ? 128 : 64;
  static constexpr int QBUF = (PAIR ? 1 : 2) * kN * 128;       // [16 rows][D], 64-wide blocks
  static constexpr int PBUF = 2 * NPV * 128;                   // [NPV rows][128 MMA rows]
  static constexpr int NPB = PAIR && G > 4 ? 1 : 2;            // P buffers that fit
  static constexpr int LENS_CAP = PAIR ? 512 : 2048;           // sequence lengths mirrored in shared memory
  static constexpr int OFF_KV = 0;
  static constexpr int OFF_Q = OFF_KV + kNS * kStage;
  static constexpr int OFF_P = OFF_Q + 2 * QBUF;
  static constexpr int OFF_RED = OFF_P + NPB * PBUF;           // [2][16][4] warp maxima, [4][16] warp sums
  static constexpr int OFF_MS = OFF_RED + (2 * 64 + 64) * 4;
  static constexpr int MS_FLOATS = 1024;                       // merge scratch; the odd keys' O at d_head 64
  static constexpr int OFF_BAR = OFF_MS + MS_FLOATS * 4;
  static constexpr int NBAR = 3 * kNS + 2 + 2 + 2 + 2 + 1 + 1;
  static constexpr int OFF_MISC = OFF_BAR + NBAR * 8;
  static constexpr int OFF_LENS = OFF_MISC + 64;
  static constexpr int RECV = dec::kClusterItems * 4 + dec::recv_floats(G, D) * 4;
  static constexpr int SMEM = OFF_LENS + cmax(LENS_CAP * 4, RECV) + 1024;
  static constexpr uint32_t IDESC_S = idesc_bf16(kBN, kN, false, false);
  static constexpr uint32_t IDESC_PV = idesc_bf16(128, NPV, false, true);
  static_assert(SMEM <= 232448, "shared memory");
  static_assert(OFF_Q % 1024 == 0 && OFF_P % 1024 == 0 && PBUF % 1024 == 0, "operand alignment");
  static_assert(OCOL + NPV <= TMEM_COLS, "TMEM columns");
  static_assert(!PAIR || G * 64 <= MS_FLOATS, "exchange of the odd keys' O");
};

// Variants of the kernel: the stream-K split; the reuse step's, with gather
// warps; and the split by whole clusters (short steps of few items).
constexpr int kStream = 0;
constexpr int kGather = 1;
constexpr int kCluster = 2;

// Gather warps of the H2Share reuse variant (warps 6 on). The cp.async
// copies a warp keeps in flight are bounded per warp, so the gather rate
// grows with the warps that issue them: sixteen for groups of up to four
// heads (704 threads, 80 registers each), eight above, where the wider
// group's softmax state needs more registers per thread.
__host__ __device__ constexpr int gather_warps(int G, int mode) {
  return mode == kGather ? (G <= 4 ? 16 : 8) : 0;
}
static_assert((kThreads + 32 * 16) * 8 <= kNS * kStage, "scan scratch");

// The items of a CTA's range, in order: next() moves to the next item that the
// CTA holds rows [sp.lo, sp.hi) of, whose first unit is item_off.
template <bool CLUSTER>
struct Walk {
  const DecodeArgs& a;
  const int* ls;
  const int n_items;
  const long long start, end;
  long long off, item_off = 0;
  int id;
  dec::Span sp;
  __device__ __forceinline__ Walk(const DecodeArgs& a_, const int* ls_, int n, long long s, long long e, int first,
                                  long long first_off, const int*)
      : a(a_), ls(ls_), n_items(n), start(s), end(e), off(first_off), id(first - 1) {}
  __device__ __forceinline__ bool next() {
    for (++id; id < n_items && off < end; ++id) {
      sp = dec::item_span(a, id, ls, off, start, end);
      item_off = off;
      off += sp.units;
      if (sp.lo < sp.hi) return true;
    }
    return false;
  }
  __device__ __forceinline__ int keys() const { return sp.keys; }
  __device__ __forceinline__ int seq(int HK) const { return id / HK; }
  // another item of the range may follow: it starts at its row 0
  __device__ __forceinline__ bool more() const { return off < end && id + 1 < n_items; }
};
// In the cluster split a CTA holds rows of one item at most (dec::plan_clusters).
template <>
struct Walk<true> {
  int id, b;
  bool left;
  long long item_off = 0;
  dec::Span sp;
  __device__ __forceinline__ Walk(const DecodeArgs&, const int*, int, long long, long long, int first, long long,
                                  const int* plan)
      : id(first), b(plan[dec::kPlanSeq]) {
    sp.keys = plan[dec::kPlanKeys];
    sp.lo = plan[dec::kPlanLo];
    sp.hi = plan[dec::kPlanHi];
    left = sp.lo < sp.hi;
  }
  __device__ __forceinline__ bool next() {
    const bool r = left;
    left = false;
    return r;
  }
  __device__ __forceinline__ int keys() const { return sp.keys; }
  __device__ __forceinline__ int seq(int) const { return b; }
  __device__ __forceinline__ bool more() const { return false; }
};

// MODE kGather: the H2Share reuse variant, whose gather warps copy the borrowed
// rows of retrieval items (a.idx != nullptr); the producer warp then loads
// only the contiguous (streaming) tiles.
// MODE kCluster: the CTAs of a cluster share one item (dec::plan_clusters) and
// add up their states through distributed shared memory
// (dec::cluster_finish); see decode_tc_cluster.cu.
template <int D, int G, int MODE>
__global__ void __launch_bounds__(kThreads + 32 * gather_warps(G, MODE), 1)
    decode_tc_kernel(const __grid_constant__ DecodeArgs a) {
  constexpr bool GATHER = MODE == kGather, CLUSTER = MODE == kCluster;
  using C = Lay<D, G>;
  constexpr bool PAIR = C::PAIR;
  constexpr int NK = C::NK;
  static_assert(!(GATHER && PAIR), "borrowed rows of d_head 64 run on the CUDA cores");
  static_assert(G >= 1 && G <= kN, "group size");
  constexpr int GW = gather_warps(G, MODE);
  constexpr int RPW = GATHER ? kBN / GW : kBN;  // rows of each tile a gather warp copies
  constexpr int NT = kThreads + 32 * GW;
  static_assert(2 * (dec::kGroup + 8) * G + 2 * G <= C::MS_FLOATS, "merge scratch");
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = smem_raw + ((1024 - (smem_u32(smem_raw) & 1023)) & 1023);
  uint8_t* sKV = smem + C::OFF_KV;
  uint8_t* sQ = smem + C::OFF_Q;
  uint8_t* sP = smem + C::OFF_P;
  float* red = reinterpret_cast<float*>(smem + C::OFF_RED);  // [2][16][4]
  float* lsum = red + 2 * 64;                             // [4][16]
  float* ms = reinterpret_cast<float*>(smem + C::OFF_MS);
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + C::OFF_BAR);  // [kNS] a TMA-loaded tile landed
  uint64_t* empty = full + kNS;
  uint64_t* gfull = empty + kNS;    // [kNS] a gathered tile landed (reuse variant)
  uint64_t* s_full = gfull + kNS;   // [2] S(j) in TMEM
  uint64_t* s_free = s_full + 2;    // [2] S(j) read by the softmax
  uint64_t* p_full = s_free + 2;    // [2] P(j) written
  uint64_t* p_free = p_full + 2;    // [2] O += P(j) V(j) done
  uint64_t* o_free = p_free + 2;    // the item's final O read
  uint64_t* drain = o_free + 1;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + C::OFF_MISC);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  long long* sh64 = reinterpret_cast<long long*>(smem + C::OFF_MISC + 8);  // [0] total, [1] first offset
  int* sh32 = reinterpret_cast<int*>(sh64 + 2);                         // [0] first item, [1] merge flag
  int* lens_s = reinterpret_cast<int*>(smem + C::OFF_LENS);
  // cluster split: the states of the cluster's CTAs for this CTA's share of the output
  float* recv = reinterpret_cast<float*>(smem + C::OFF_LENS + dec::kClusterItems * 4);

  const CacheGeom& g = a.geom;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int HK = g.n_r + g.n_s;
  const int n_items = g.B * HK;
  const int P = a.n_ctas, p = blockIdx.x;

  // Prologue that touches no global memory; it may overlap the tail of the
  // previous kernel on the stream (programmatic dependent launch).
  // Q and P rows >= G stay zero for the whole launch
  for (int i = threadIdx.x; i < (2 * C::QBUF + C::NPB * C::PBUF) / 16; i += NT)
    reinterpret_cast<uint4*>(sQ)[i] = make_uint4(0, 0, 0, 0);
  fence_proxy_async_smem();
  if (threadIdx.x == 0) {
    for (int s = 0; s < kNS; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
      mbar_init(&gfull[s], GATHER ? GW : 1);
    }
    for (int x = 0; x < 2; ++x) {
      mbar_init(&s_full[x], 1);
      mbar_init(&s_free[x], 4);
      mbar_init(&p_full[x], 4);
      mbar_init(&p_free[x], 1);
    }
    mbar_init(o_free, 4);
    mbar_init(drain, 1);
    *abort_flag = 0;
    fence_mbar_init();
  }
  if (warp == 4 && lane == 0) {
    if (g.n_r > 0) prefetch_tmap(&a.tcr);
    if (g.n_s > 0) prefetch_tmap(&a.tcs);
    if (PAIR && g.n_r > 0) prefetch_tmap(&a.tcr_odd);
    if (PAIR && g.n_s > 0) prefetch_tmap(&a.tcs_odd);
  }
  if (warp == 5) {
    tmem_alloc(tmem_slot, C::TMEM_COLS);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  const dec::PlanSetup plan_setup(g);
  // a CTA writes into its cluster's shared memory only once every CTA of it runs
  if constexpr (CLUSTER) cluster_arrive();
  // everything the previous kernels wrote (lengths, cache, inputs, counters)
  // is visible after this wait; the next step may then start its prologue
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  // the lengths do not change before every CTA has this copy, which all roles
  // read (the last CTA to finish, or on the cluster split to have issued its
  // copies, advances them)
  const int* ls = g.B <= C::LENS_CAP ? lens_s : nullptr;
  if (!CLUSTER && ls != nullptr) {  // plan_clusters does it
    for (int i = threadIdx.x; i < g.B; i += NT) lens_s[i] = __ldcg(&a.lens[i]);
    __syncthreads();
  }
  long long total = 0, start = 0, end = 0, first_off = 0;
  if constexpr (CLUSTER) {
    // the producer plans, and goes on to its copies without a block barrier
    if (warp == 4) {
      dec::plan_clusters(a, plan_setup, lens_s, kBN, sh32);
      __syncwarp();
      named_barrier_arrive(2, NT);
    } else {
      named_barrier_sync(2, NT);
    }
    cluster_wait();
  } else {
    dec::find_cta_range<NT>(a, reinterpret_cast<long long*>(sKV), sh64, sh32, ls);
    __syncthreads();
    total = sh64[0];
    start = (long long)p * total / P;
    end = (long long)(p + 1) * total / P;
    first_off = sh64[1];
  }
  const int first_id = sh32[0];
  Walk<CLUSTER> walk(a, ls, n_items, start, end, first_id, first_off, sh32);

  if (warp == 4) {
    // ------------------------------------------------------------ producer
    // Lane 0 loads 128-row K and V tiles of the region (4D tensor maps over
    // the cache regions, 128-byte swizzle). In the reuse variant the gather
    // warps issue every tile instead (see below) and this warp idles.
    if (!GATHER && lane == 0) {
      int it = 0;
      bool ok = true;
      while (ok && walk.next()) {
        const int id = walk.id, lo = walk.sp.lo, hi = walk.sp.hi;
        const int b = walk.seq(HK), k = id - b * HK;
        const bool strm = k >= g.n_r;
        const int region = strm ? b * g.n_s + (k - g.n_r) : b * g.n_r + k;
        const CUtensorMap* map = strm ? &a.tcs : &a.tcr;
        const CUtensorMap* map_odd = strm ? &a.tcs_odd : &a.tcr_odd;
        for (int row0 = lo; row0 < hi; row0 += kBN, ++it) {
          const int st = it % kNS;
          if (it >= kNS && !wait_bar(&empty[st], ((it / kNS) & 1) ^ 1, a.err, abort_flag)) {
            ok = false;
            break;
          }
          mbar_arrive_expect_tx(&full[st], kStage);
          uint8_t* dst = sKV + st * kStage;
#pragma unroll
          for (int sel = 0; sel < 2; ++sel)
#pragma unroll
            for (int db = 0; db < 2; ++db)
              tma_load_4d(dst + sel * kTile + db * kBox, PAIR && db == 1 ? map_odd : map, PAIR ? 0 : db * 64, row0,
                          sel, region, &full[st]);
        }
      }
      if constexpr (CLUSTER) dec::advance_lens(a, lens_s);
      // every issued copy lands before the CTA can exit
      for (int j = it > kNS ? it - kNS : 0; j < it; ++j) drain_wait(&full[j % kNS], (j / kNS) & 1, a.err);
    }
    __syncwarp();
  } else if (GATHER && warp >= 6) {
    // ------------------------------------------------------------ gatherers
    // The reuse variant's GW gather warps issue every tile of the CTA's
    // range, each of them waiting for every tile's stage to be free, in
    // order (an mbarrier parity wait is only sound within one phase of the
    // barrier, so no waiter may skip tiles). Contiguous (streaming) tiles:
    // lane 0 of warp 6 loads them with the TMA onto full[st]. Retrieval
    // items: gather warp w copies rows RPW w .. RPW w + RPW - 1 of each
    // 128-row tile of borrowed positions, one row per instruction (lanes
    // 0-15 the 16 chunks of its K row, lanes 16-31 those of its V row) with
    // 16-byte cp.async copies into the swizzled layout the MMAs read, and the
    // copies complete on gfull[st]; the new token's row (position t, not in
    // the cache yet) comes from the step's input. Lane j < RPW holds the
    // index of row RPW w + j, loaded two tiles ahead into one of two
    // registers that alternate between tiles (a register copy of an
    // in-flight load would wait for it). Row gathers through the TMA
    // (tile::gather4 or bulk row copies) ran at about 15 GB/s per SM;
    // cp.async copies scale with the issuing warps.
    const int gw = warp - 6;
    const int half = lane >> 4, ch = lane & 15;
    const uint32_t dst_lane = half * kTile + (ch >> 3) * kBox;
    const uint32_t swz = ch & 7;
    const bool loader = gw == 0 && lane == 0;  // issues the TMA tiles
    int it = 0;
    bool ok = true;
    uint32_t fpar = 0;  // loader: bit st, parity of stage st's next full[] phase
    uint32_t mine = 0;  // loader: bit st, stage st's latest tile came through the TMA
    auto stage_free = [&](int st) -> bool {  // warp-uniform
      int go = 1;
      if (lane == 0 && it >= kNS && !wait_bar(&empty[st], ((it / kNS) & 1) ^ 1, a.err, abort_flag)) go = 0;
      return __shfl_sync(0xffffffffu, go, 0) != 0;
    };
    while (ok && walk.next()) {
      const int id = walk.id, lo = walk.sp.lo, hi = walk.sp.hi;
      const int b = walk.seq(HK), k = id - b * HK;
      if (k >= g.n_r) {
        const int region = b * g.n_s + (k - g.n_r);
        for (int row0 = lo; row0 < hi; row0 += kBN, ++it) {
          const int st = it % kNS;
          if (!stage_free(st)) {
            ok = false;
            break;
          }
          if (loader) {
            mbar_arrive_expect_tx(&full[st], kStage);
            uint8_t* dst = sKV + st * kStage;
#pragma unroll
            for (int sel = 0; sel < 2; ++sel)
#pragma unroll
              for (int db = 0; db < 2; ++db)
                tma_load_4d(dst + sel * kTile + db * kBox, &a.tcs, db * 64, row0, sel, region, &full[st]);
            fpar ^= 1u << st;
            mine |= 1u << st;
          }
        }
        continue;
      }
      const int32_t* rowlist = a.idx + ((size_t)b * a.n_idx_groups + a.idx_map[k]) * a.top_k;
      const int t = dec::seq_len(a, b, ls);
      const bf16* src_base =
          static_cast<const bf16*>(a.kv) + g.r_region(b, k) + (half ? (size_t)g.max_seq * D : 0) + ch * 8;
      const bf16* src_new =
          static_cast<const bf16*>(half ? a.v_new : a.k_new) + ((size_t)b * g.Hkv + g.r_head[k]) * D + ch * 8;
      const bool idx_lane = lane < RPW;
      const int j0 = lo + RPW * gw + lane;
      int ia = idx_lane && j0 < hi ? __ldg(rowlist + j0) : 0;
      int ib = idx_lane && j0 + kBN < hi ? __ldg(rowlist + j0 + kBN) : 0;
      auto gather_tile = [&](int row0, int& buf) -> bool {
        const int my_row = idx_lane && row0 + RPW * gw + lane < hi ? min(max(buf, 0), t) : -1;
        const int jn = row0 + 2 * kBN + RPW * gw + lane;
        buf = idx_lane && jn < hi ? __ldg(rowlist + jn) : 0;
        const int st = it % kNS;
        if (!stage_free(st)) return false;
        uint8_t* tile = sKV + st * kStage + dst_lane;
#pragma unroll 8
        for (int j = 0; j < RPW; ++j) {
          const int c = __shfl_sync(0xffffffffu, my_row, j);
          const int r = RPW * gw + j;
          if (c >= 0)
            cp_async16(tile + r * 128 + ((swz ^ (uint32_t)(r & 7)) << 4),
                       c == t ? src_new : src_base + (size_t)c * D);
        }
        cp_async_mbar_arrive(&gfull[st]);
        __syncwarp();
        if (lane == 0) mbar_arrive(&gfull[st]);
        if (loader) mine &= ~(1u << st);
        ++it;
        return true;
      };
      for (int row0 = lo; row0 < hi; row0 += 2 * kBN) {
        if (!gather_tile(row0, ia)) {
          ok = false;
          break;
        }
        if (row0 + kBN >= hi) break;
        if (!gather_tile(row0 + kBN, ib)) {
          ok = false;
          break;
        }
      }
    }
    // every copy issued here lands before the CTA can exit: the cp.async
    // copies, and the latest TMA tile of each stage
    asm volatile("cp.async.wait_all;" ::: "memory");
    if (loader)
      for (int st = 0; st < kNS; ++st)
        if (mine & (1u << st)) drain_wait(&full[st], ((fpar >> st) & 1) ^ 1, a.err);
    __syncwarp();
  } else if (warp == 5) {
    // ------------------------------------------------------------ MMA issuer
    const uint64_t k_desc0 = sdesc_sw128(smem_u32(sKV), 16, 1024);
    const uint64_t v_desc0 = sdesc_sw128(smem_u32(sKV) + kTile, kBox, 1024);
    const uint64_t q_desc0 = sdesc_sw128(smem_u32(sQ), 16, 1024), p_desc0 = sdesc_sw128(smem_u32(sP), 16, 1024);
    int it = 0, item_k = 0, ofw = 0;
    uint32_t fpar = 0, gpar = 0;  // bit st: parity of stage st's next full[] / gfull[] phase
    bool ok = true;
    struct Pend {
      int it, st, item;
      bool first;
    } pend{0, 0, 0, false};
    bool has_pend = false;
    auto wait_warp = [&](uint64_t* bar, uint32_t parity) {
      if (ok) ok = __all_sync(0xffffffffu, wait_bar(bar, parity, a.err, abort_flag));
    };
    // o_free phases complete once per item, in order
    auto wait_ofree = [&](int n) {
      while (ok && ofw < n) {
        wait_warp(o_free, ofw & 1);
        ++ofw;
      }
    };
    auto issue_pv = [&](const Pend& t) {
      wait_warp(&p_full[t.it & 1], (t.it >> 1) & 1);
      if (t.first && t.item >= 1) wait_ofree(t.item);  // accumulate = 0 overwrites the last item's O
      if (!ok) return;
      if (elect_one()) {
        tc_fence_after();
        const uint64_t v_desc = v_desc0 + (uint32_t)(t.st * sdesc_step(kStage));
        const uint64_t p_desc = p_desc0 + (uint32_t)((t.it % C::NPB) * sdesc_step(C::PBUF));
#pragma unroll
        for (int kk = 0; kk < kBN / 16; ++kk) {
          const uint64_t ad = v_desc + sdesc_step(kk * 2048);
          const uint64_t bd = p_desc + sdesc_step((kk >> 2) * (C::NPV * 128) + (kk & 3) * 32);
          tc_mma(tmem + C::OCOL, ad, bd, C::IDESC_PV, (t.first && kk == 0) ? 0u : 1u);
        }
        tc_commit(&p_free[t.it & 1]);
        tc_commit(&empty[t.st]);
      }
      __syncwarp();
    };

    // An item's global inputs (its G query rows; the new token's K and V
    // row) are fetched into registers one item ahead: under the saturated
    // HBM stream a plain load takes microseconds, which at an item switch
    // would sit between this item's last P V and the next item's first S.
    // Lane l holds 16-byte chunks l, l + 32, ... of the G x D query block (CPR
    // chunks a head); lanes 0 .. CPR - 1 the new K row's chunks, the next CPR
    // lanes the new V row's.
    constexpr int CPR = D / 8;
    constexpr int QV = (G * CPR + 31) / 32;
    uint4 qr[QV];
    uint4 nvr;
    const int ch = lane % CPR;
    const bool new_v = lane >= CPR, new_lane = lane < 2 * CPR;
    auto fetch_inputs = [&](int id) {
      const int b = CLUSTER ? walk.seq(HK) : id / HK, k = id - b * HK;
      const int kvh = k >= g.n_r ? (int)g.s_head[k - g.n_r] : (int)g.r_head[k];
      const bf16* qg = static_cast<const bf16*>(a.q) + ((size_t)b * g.Hq + (size_t)kvh * G) * D;
#pragma unroll
      for (int i = 0; i < QV; ++i) {
        const int c = lane + 32 * i;
        if (c < G * CPR) qr[i] = *reinterpret_cast<const uint4*>(qg + (size_t)(c / CPR) * D + (c % CPR) * 8);
      }
      const size_t new_off = ((size_t)b * g.Hkv + kvh) * D + ch * 8;
      nvr = *reinterpret_cast<const uint4*>(static_cast<const bf16*>(new_v ? a.v_new : a.k_new) + new_off);
    };
    int fetched = -1;  // the item whose inputs the registers hold
    if (first_id < n_items) {
      fetch_inputs(first_id);
      fetched = first_id;
    }

    while (ok && walk.next()) {
      const int id = walk.id, lo = walk.sp.lo, hi = walk.sp.hi;
      const int b = walk.seq(HK), k = id - b * HK;
      const bool strm = k >= g.n_r;
      const int hi_idx = strm ? k - g.n_r : k;
      const int t = dec::seq_len(a, b, ls);
      const int cap = strm ? g.S + g.W : g.max_seq;
      const int xr = strm ? (t < g.S ? t : g.S + (t - g.S) % g.W) : t;  // the new token's row
      bf16* Kc = static_cast<bf16*>(a.kv) + (strm ? g.s_region(b, hi_idx) : g.r_region(b, hi_idx));
      bf16* Vc = Kc + (size_t)cap * D;

      // this item's Q into buffer item_k & 1, last read by the MMAs of item item_k - 2
      wait_ofree(item_k - 1);
      if (!ok) break;
      if (fetched != id) {  // an item skipped by this CTA took the prefetch
        fetch_inputs(id);
        fetched = id;
      }
      {
        uint8_t* qs = sQ + (item_k & 1) * C::QBUF;
#pragma unroll
        for (int i = 0; i < QV; ++i) {
          const int c = lane + 32 * i;
          if (c < G * CPR) {
            const int h = c / CPR, cc = c % CPR;
            *reinterpret_cast<uint4*>(qs + (cc >> 3) * (kN * 128) + h * 128 + (((cc & 7) ^ (h & 7)) << 4)) = qr[i];
          }
        }
        fence_proxy_async_smem();
        __syncwarp();
      }
      const uint4 nv = nvr;
      // the next item of this CTA's range starts at its row 0
      if (walk.more()) {
        fetch_inputs(id + 1);
        fetched = id + 1;
      }

      // H2Share reuse step: this retrieval item's rows are gathered
      const bool gathered = GATHER && a.idx != nullptr && !strm;
      for (int row0 = lo; row0 < hi; row0 += kBN, ++it) {
        const int st = it % kNS;
        const int cnt = min(kBN, hi - row0);
        // a tile landed on full[st] (TMA) or gfull[st] (gather warps)
        wait_warp(gathered ? &gfull[st] : &full[st], ((gathered ? gpar : fpar) >> st) & 1);
        if (gathered)
          gpar ^= 1u << st;
        else
          fpar ^= 1u << st;
        if (!ok) break;
        auto put_new_row = [&](int r) {  // the new token's K / V chunk into tile row r
          const int box = PAIR ? xr & 1 : ch >> 3;
          uint8_t* dst =
              sKV + st * kStage + (new_v ? kTile : 0) + box * kBox + r * 128 + (((ch & 7) ^ (r & 7)) << 4);
          *reinterpret_cast<uint4*>(dst) = nv;
        };
        if (gathered) {
          // the gather warps wrote this tile with cp.async (generic proxy):
          // order it before the tensor core's reads; the item's owner of row
          // 0 appends the new token
          if (row0 == 0) *reinterpret_cast<uint4*>((new_v ? Vc : Kc) + (size_t)xr * D + ch * 8) = nv;
          fence_proxy_async_smem();
          __syncwarp();
        } else if (xr / NK >= row0 && xr / NK < row0 + cnt) {
          if (new_lane) {
            put_new_row(xr / NK - row0);
            *reinterpret_cast<uint4*>((new_v ? Vc : Kc) + (size_t)xr * D + ch * 8) = nv;  // append
          }
          fence_proxy_async_smem();
          __syncwarp();
        }
        if (it >= 2) wait_warp(&s_free[it & 1], ((it >> 1) - 1) & 1);
        if (!ok) break;
        if (elect_one()) {
          tc_fence_after();
          const uint64_t k_desc = k_desc0 + (uint32_t)(st * sdesc_step(kStage));
          const uint64_t q_desc = q_desc0 + (uint32_t)((item_k & 1) * sdesc_step(C::QBUF));
#pragma unroll
          for (int kk = 0; kk < 8; ++kk) {
            // d_head 128: 8 K-steps over both blocks; 64: 4 over each parity's block
            const int y = PAIR ? kk >> 2 : 0;
            const uint64_t ad = k_desc + sdesc_step((kk >> 2) * kBox + (kk & 3) * 32);
            const uint64_t bd = q_desc + sdesc_step((PAIR ? 0 : kk >> 2) * (kN * 128) + (kk & 3) * 32);
            tc_mma(tmem + (it & 1) * C::SCOLS + y * kN, ad, bd, C::IDESC_S, (PAIR ? kk & 3 : kk) > 0 ? 1u : 0u);
          }
          tc_commit(&s_full[it & 1]);
        }
        __syncwarp();
        if (has_pend) issue_pv(pend);
        pend = Pend{it, st, item_k, row0 == lo};
        has_pend = true;
        if (gathered) {
          // a gathered tile's P V goes out as soon as its P is written:
          // the next tile arrives late (random rows), and its stage is
          // freed only by this P V
          issue_pv(pend);
          has_pend = false;
        }
      }
      // Inside an item, P(j) V(j) waits behind S(j + 1) so that the softmax
      // of tile j + 1 can start meanwhile. At the item's end nothing can
      // use the next item's S before this item's O is final, and holding
      // P V back until the next item's first tile lands (a loaded-DRAM
      // round trip) would hold the epilogue and this tile's ring slot.
      if (has_pend && ok) {
        issue_pv(pend);
        has_pend = false;
      }
      ++item_k;
    }
    if (has_pend) issue_pv(pend);
    if (elect_one()) tc_commit(drain);
    __syncwarp();
    drain_wait(drain, 0, a.err);
    __syncwarp();
  } else {
    // ------------------------------------------------------------ softmax
    const int t = threadIdx.x;  // key of the tile / row d of O^T
    const uint32_t tl = tmem + ((uint32_t)(warp * 32) << 16);
    int it = 0;
    // ok: the four warps' common verdict, only ever set at a barrier (so every
    // thread leaves the loops together); local_ok: this thread's waits since
    bool ok = true, local_ok = true;
    uint32_t fpar = 0, gpar = 0;  // bit st: parity of stage st's next full[] / gfull[] phase
    if constexpr (CLUSTER) {
      if (!walk.left) dec::cluster_push_empty<G, D>(recv);
    }
    while (ok && walk.next()) {
      const int id = walk.id, lo = walk.sp.lo, hi = walk.sp.hi;
      const int b = walk.seq(HK), k = id - b * HK;
      const bool strm = k >= g.n_r;
      const int kvh = strm ? g.s_head[k - g.n_r] : g.r_head[k];

      float m[G], l[G];
#pragma unroll
      for (int h = 0; h < G; ++h) {
        m[h] = -INFINITY;
        l[h] = 0.f;
      }
      const bool gathered = GATHER && a.idx != nullptr && !strm;
      for (int row0 = lo; row0 < hi; row0 += kBN, ++it) {
        const int x = it & 1, st = it % kNS;
        const int cnt = min(kBN, hi - row0);
        const uint32_t land_par = ((gathered ? gpar : fpar) >> st) & 1;  // the phase that lands this tile
        if (gathered)
          gpar ^= 1u << st;
        else
          fpar ^= 1u << st;
        // the tile's keys that the item holds (at d_head 64 the last pair may hold one)
        const int kv = PAIR ? min(2 * cnt, walk.keys() - 2 * row0) : cnt;
        if (kv < NK * kBN) {
          // zero the V rows of this warp's keys that the item does not hold (d_head
          // 128: both halves) while S is formed. The lanes' chunks lie side by
          // side: each lane zeroing its own row met bank conflicts, 2,100 clocks at
          // a step's last tile, and after S the rest, 500, still held up the step
          local_ok = wait_bar(gathered ? &gfull[st] : &full[st], land_par, a.err, abort_flag) && local_ok;
          const int end = (warp + 1) * 32;
#pragma unroll
          for (int box = 0; box < 2; ++box) {
            const int first = max(warp * 32, PAIR ? (kv + 1 - box) / 2 : kv);  // first row to zero
            uint4* v4 = reinterpret_cast<uint4*>(sKV + st * kStage + kTile + box * kBox);
            for (int c = first * 8 + lane; c < end * 8; c += 32) v4[c] = make_uint4(0, 0, 0, 0);
          }
        }
        local_ok = wait_bar(&s_full[x], (it >> 1) & 1, a.err, abort_flag) && local_ok;
        tc_fence_after();
        uint32_t v[NK][PAIR ? 8 : 16];
        if constexpr (PAIR) {
          tmem_ld8(tl + x * C::SCOLS, v[0]);
          tmem_ld8(tl + x * C::SCOLS + kN, v[1]);
        } else {
          tmem_ld16(tl + x * C::SCOLS, v[0]);
        }
        tmem_ld_wait();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&s_free[x]);
        bool valid[NK];
        float s[NK][G];
#pragma unroll
        for (int y = 0; y < NK; ++y) {
          valid[y] = NK * t + y < kv;
#pragma unroll
          for (int h = 0; h < G; ++h) s[y][h] = valid[y] ? __uint_as_float(v[y][h]) * a.scale_log2 : -INFINITY;
        }
        if (!PAIR && a.scores != nullptr && !strm && valid[0]) {
          // H2Share anchor step: this row's scores for the top-k selection
          float* sc = a.scores + ((size_t)(b * g.n_r + k) * G) * a.score_stride + row0 + t;
#pragma unroll
          for (int h = 0; h < G; ++h) sc[(size_t)h * a.score_stride] = s[0][h];
        }

        // per-head maximum over the tile: each warp, then the four warps
        float* rx = red + x * 64;
        float wm = -INFINITY;
#pragma unroll
        for (int h = 0; h < G; ++h) {
          const float r = warp_max(PAIR ? fmaxf(s[0][h], s[NK - 1][h]) : s[0][h]);
          wm = (lane == h) ? r : wm;
        }
        if (lane < G) rx[lane * 4 + warp] = wm;
        ok = named_barrier_and(1, kSoftmaxThreads, local_ok);
        if (!ok) break;
        // one 16-byte load a head, and a single uniform branch past the first tile
        bool resc = false;
        float alpha[G], tm[G];
#pragma unroll
        for (int h = 0; h < G; ++h) {
          const float4 w4 = *reinterpret_cast<const float4*>(rx + h * 4);
          tm[h] = fmaxf(fmax3f(w4.x, w4.y, w4.z), w4.w);
          alpha[h] = 1.f;
          if (row0 == lo)
            m[h] = fmaxf(m[h], tm[h]);
          else
            resc = resc || tm[h] > m[h] + kRescaleThreshold;
        }
        if (resc) {
#pragma unroll
          for (int h = 0; h < G; ++h) {
            if (tm[h] > m[h] + kRescaleThreshold) {
              alpha[h] = (m[h] == -INFINITY) ? 0.f : fast_exp2(m[h] - tm[h]);
              m[h] = tm[h];
              l[h] *= alpha[h];
            }
          }
        }
        // the P buffer is free once O += P(it - NPB) V is done
        if (it >= C::NPB)
          local_ok = wait_bar(&p_free[(it - C::NPB) & 1], ((it - C::NPB) >> 1) & 1, a.err, abort_flag) && local_ok;
        if (resc) {
          // rescale row t of O^T; O += P(it - 1) V must have landed first
          local_ok = wait_bar(&p_free[x ^ 1], ((it - 1) >> 1) & 1, a.err, abort_flag) && local_ok;
          tc_fence_after();
          uint32_t o[C::NP];
#pragma unroll
          for (int q = 0; q < C::PARTS; ++q) {
            tmem_ld(tl + C::OCOL + q * C::NP, o);
            tmem_ld_wait();
#pragma unroll
            for (int c = 0; c < C::NP; ++c)
              if (c % C::HP < G) o[c] = __float_as_uint(__uint_as_float(o[c]) * alpha[c % C::HP]);
            tmem_st(tl + C::OCOL + q * C::NP, o);
          }
          tmem_st_wait();
        }
        float pr[NK][G];
#pragma unroll
        for (int y = 0; y < NK; ++y)
#pragma unroll
          for (int h = 0; h < G; ++h) {
            pr[y][h] = valid[y] ? fast_exp2(s[y][h] - m[h]) : 0.f;
            l[h] += pr[y][h];
          }
        // P^T row t -> column t of the K-major [NPV][128 rows] buffer
        uint8_t* pb = sP + (it % C::NPB) * C::PBUF + (t >> 6) * (C::NPV * 128) + (t & 7) * 2;
        const int j = (t & 63) >> 3;
#pragma unroll
        for (int y = 0; y < NK; ++y)
#pragma unroll
          for (int h = 0; h < G; ++h) {
            float rest = pr[y][h];
#pragma unroll
            for (int q = 0; q < C::PARTS; ++q) {
              const int n = q * C::NP + y * C::HP + h;
              const bf16 part = __float2bfloat16_rn(rest);
              *reinterpret_cast<bf16*>(pb + n * 128 + ((j ^ (n & 7)) << 4)) = part;
              rest -= __bfloat162float(part);
            }
          }
        fence_proxy_async_smem();
        tc_fence_before();
        __syncwarp();
        if (lane == 0 && !(it == 0 && p == a.stall_cta)) mbar_arrive(&p_full[x]);
      }
      if (!ok) break;

      // ---- the item's state: O^T row t, m (uniform), l summed over the keys (while
      // the last P V runs)
#pragma unroll
      for (int h = 0; h < G; ++h) {
        float v = l[h];
#pragma unroll
        for (int msk = 16; msk >= 1; msk >>= 1) v += __shfl_xor_sync(0xffffffffu, v, msk);
        if (lane == 0) lsum[warp * 16 + h] = v;
      }
      const int last = it - 1;
      local_ok = wait_bar(&p_free[last & 1], (last >> 1) & 1, a.err, abort_flag) && local_ok;
      tc_fence_after();
      uint32_t o[C::NP];
      tmem_ld(tl + C::OCOL, o);
      if constexpr (PAIR) {
        uint32_t o1[C::NP], o2[C::NP];
        tmem_ld(tl + C::OCOL + C::NP, o1);
        tmem_ld(tl + C::OCOL + 2 * C::NP, o2);
        tmem_ld_wait();
        // an infinite V row makes the first sum infinite and the others NaN where a
        // part of its weight is zero: the first sum is the result then
#pragma unroll
        for (int c = 0; c < C::NP; ++c) {
          const float s = __uint_as_float(o[c]);
          if (!isinf(s)) o[c] = __float_as_uint(s + (__uint_as_float(o1[c]) + __uint_as_float(o2[c])));
        }
      } else {
        tmem_ld_wait();
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(o_free);
      if (PAIR && t >= 64) {
#pragma unroll
        for (int h = 0; h < G; ++h) ms[h * 64 + t - 64] = __uint_as_float(o[NK * C::HP - C::HP + h]);
      }
      ok = named_barrier_and(1, kSoftmaxThreads, local_ok);
      if (!ok) break;
      if (PAIR && t < 64) {
#pragma unroll
        for (int h = 0; h < G; ++h) o[h] = __float_as_uint(__uint_as_float(o[h]) + ms[h * 64 + t]);
      }
      const bool row_d = t < D;  // this thread holds row d = t of the result
      float L[G];
#pragma unroll
      for (int h = 0; h < G; ++h) L[h] = (lsum[h] + lsum[16 + h]) + (lsum[32 + h] + lsum[48 + h]);

      if constexpr (CLUSTER) {
        dec::cluster_push<G, D>(recv, o, m, L);
      } else {
        const long long row_off = walk.item_off + walk.sp.cost;  // unit of the item's row 0
        const int f = dec::cta_of(row_off, total, P);
        const int lst = dec::cta_of(row_off + (long long)(walk.sp.rows - 1) * walk.sp.w, total, P);
        bf16* outp = static_cast<bf16*>(a.out) + ((size_t)b * g.Hq + (size_t)kvh * G) * D;
        float2* st = (a.scores != nullptr && !strm) ? a.score_stats + (size_t)(b * g.n_r + k) * G : nullptr;
        if (f == lst) {
#pragma unroll
          for (int h = 0; h < G; ++h)
            if (row_d) outp[h * D + t] = __float2bfloat16_rn(__uint_as_float(o[h]) / L[h]);
          if (st != nullptr && t < G) {
            float mt = m[0], lt = L[0];
#pragma unroll
            for (int h = 1; h < G; ++h) {
              mt = (t == h) ? m[h] : mt;
              lt = (t == h) ? L[h] : lt;
            }
            st[t] = make_float2(mt, lt);
          }
        } else {
          float* pbase = dec::partial_slot(a, p, p == f ? 1 : 0, G, D);
#pragma unroll
          for (int h = 0; h < G; ++h)
            if (row_d) __stcg(pbase + h * D + t, __uint_as_float(o[h]));
          float mt = m[0], lt = L[0];
#pragma unroll
          for (int h = 1; h < G; ++h) {
            mt = (t == h) ? m[h] : mt;
            lt = (t == h) ? L[h] : lt;
          }
          if (t < G) {
            __stcg(pbase + G * D + t, mt);
            __stcg(pbase + G * D + G + t, lt);
          }
          dec::merge_item<G, D, kSoftmaxThreads, true>(a, p, f, lst, id, outp, ms, sh32 + 1, st);
        }
        named_barrier_sync(1, kSoftmaxThreads);
      }
    }
  }

  tc_fence_before();
  if constexpr (CLUSTER) {
    // every CTA's state has arrived; the waits of an aborted CTA are bounded,
    // so it comes here too
    cluster_arrive();
    const bool any = first_id < n_items;
    const int b = any ? walk.seq(HK) : 0, k = any ? first_id - b * HK : 0;
    const bool strm = k >= g.n_r;
    const int kvh = strm ? g.s_head[k - g.n_r] : g.r_head[k];
    bf16* outp = static_cast<bf16*>(a.out) + ((size_t)b * g.Hq + (size_t)kvh * G) * D;
    float2* st = (a.scores != nullptr && !strm) ? a.score_stats + (size_t)(b * g.n_r + k) * G : nullptr;
    cluster_wait();
    if (warp < 4 && any) {
      dec::cluster_finish<G, D, kSoftmaxThreads>(a, recv, sh32, outp, st);
    }
  }
  __syncthreads();
  tc_fence_after();
  if (warp == 5) tmem_dealloc(tmem, C::TMEM_COLS);
  if constexpr (!CLUSTER)
    if (threadIdx.x == 0) dec::finish_launch(a, ls);
}

// `cluster`: CTAs per cluster (kCluster; it divides a.n_ctas).
template <int D, int G, int MODE>
cudaError_t launch_g(const DecodeArgs& a, int cluster, cudaStream_t s) {
  static std::atomic<uint64_t> done{0};
  const cudaError_t e = once_per_device(done, [] {
    cudaError_t e =
        cudaFuncSetAttribute(decode_tc_kernel<D, G, MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, Lay<D, G>::SMEM);
    if (e == cudaSuccess && MODE == kCluster)
      e = cudaFuncSetAttribute(decode_tc_kernel<D, G, MODE>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    return e;
  });
  if (e != cudaSuccess) return e;
  // programmatic stream serialization: the kernel waits for the previous
  // work on the stream itself (griddepcontrol.wait) after its prologue
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(a.n_ctas);
  cfg.blockDim = dim3(kThreads + 32 * gather_warps(G, MODE));
  cfg.dynamicSmemBytes = Lay<D, G>::SMEM;
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  if (MODE == kCluster) {
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = cluster;
    attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
    cfg.numAttrs = 2;
  }
  return cudaLaunchKernelEx(&cfg, decode_tc_kernel<D, G, MODE>, a);
}

template <int D, int MODE>
cudaError_t launch_mode(const DecodeArgs& a, int cluster, cudaStream_t s) {
  switch (a.geom.G) {
    case 1: return launch_g<D, 1, MODE>(a, cluster, s);
    case 2: return launch_g<D, 2, MODE>(a, cluster, s);
    case 4: return launch_g<D, 4, MODE>(a, cluster, s);
    case 7: return launch_g<D, 7, MODE>(a, cluster, s);
    case 8: return launch_g<D, 8, MODE>(a, cluster, s);
  }
  if constexpr (D == 128) {
    switch (a.geom.G) {
      case 3: return launch_g<D, 3, MODE>(a, cluster, s);
      case 5: return launch_g<D, 5, MODE>(a, cluster, s);
      case 6: return launch_g<D, 6, MODE>(a, cluster, s);
      case 16: return launch_g<D, 16, MODE>(a, cluster, s);
    }
  }
  return cudaErrorInvalidValue;
}

}  // namespace dtc
}  // namespace aoh
