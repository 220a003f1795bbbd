// Effective-rank head classifier (Sec. 4: Eq. 2-6 and Algorithm 1; Appendix
// "GQA Extension"): exact Gram matrices from digit products on the tensor
// cores, fp64 on CUDA cores after them. It runs once per model, offline; exactness
// matters more than speed.
//
// For query head h with projections W_Q^h, W_K^h ([d_head][d_model]) the
// kernel attention matrix M_h = W_K^T W_Q (Eq. 2) has rank <= d_head, and
// its singular values are those of the d_head x d_head matrix
//   A = L_K^T L_Q,  with  W_Q W_Q^T = L_Q L_Q^T,  W_K W_K^T = L_K L_K^T
// (Cholesky factors; W^T = Q L^T is a thin QR, so M_h = Q_K (L_K^T L_Q) Q_Q^T).
// Steps:
//   1. row_exp_kernel: the scale of every weight row; gram_tc_kernel: Gram
//      matrices W W^T of every query and key projection (products and sums are
//      exact; the d_model range is split over CTAs, each part rounds once to
//      fp64, and the parts are summed in a fixed order, so the result does not
//      depend on scheduling).
//   2. chol_kernel: semi-definite Cholesky in shared memory; a pivot at or
//      below d_head * eps * max(diag) leaves a zero column (rank deficiency).
//   3. bidiag_kernel: A = L_K^T L_Q and its bidiagonal form; svals_kernel:
//      its singular values. Values at or below sigma_max * d_model * eps are
//      the zeros of a rank-deficient M_h and are dropped (Eq. 4 sums over
//      nonzero values); ER (Eq. 4) is exp of the entropy of the normalised
//      singular values.
//   4. classify_kernel: per layer, group score = mean ER of the group's
//      query heads; the k = ceil((100 - s) * groups / 100) lowest groups
//      (stable order, ties to the lower index) are retrieval, the rest
//      streaming.
// One call takes all layers of a model, so every matrix is a CTA of its own
// and the GPU fills up.
#include <float.h>
#include <math.h>

#include <algorithm>

#include "../../include/aoh.h"
#include "common.cuh"
#include "internal.h"
#include "tc.cuh"

namespace aoh {
namespace {

using bf16 = __nv_bfloat16;

// Matrices are numbered layer-major: layer l's query projections, then its
// key projections (nmat = Hq + Hkv per layer).
__device__ __forceinline__ const bf16* weight_of(const bf16* wq, const bf16* wk, int m, int Hq, int Hkv, int dh,
                                                 int dm) {
  const int nmat = Hq + Hkv, l = m / nmat, mi = m % nmat;
  return mi < Hq ? wq + ((size_t)l * Hq + mi) * dh * dm : wk + ((size_t)l * Hkv + (mi - Hq)) * dh * dm;
}

// Largest exponent field of every weight row (255: the row holds an infinity
// or a NaN), one warp per row; rows are numbered matrix-major.
__global__ void __launch_bounds__(256) row_exp_kernel(const bf16* wq, const bf16* wk, int Hq, int Hkv, int rows, int dh,
                                                      int dm, int vec, int* row_exp) {
  const int row = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (row >= rows) return;
  const uint16_t* w =
      reinterpret_cast<const uint16_t*>(weight_of(wq, wk, row / dh, Hq, Hkv, dh, dm)) + (size_t)(row % dh) * dm;
  uint32_t m = 0;  // the largest magnitude, two halves a word when vec
  if (vec) {
    for (int c = lane; c < dm / 8; c += 32) {
      const uint4 v = __ldg(reinterpret_cast<const uint4*>(w) + c);
      m = __vmaxu2(m, __vmaxu2(__vmaxu2(v.x & 0x7fff7fffu, v.y & 0x7fff7fffu),
                               __vmaxu2(v.z & 0x7fff7fffu, v.w & 0x7fff7fffu)));
    }
  } else {
    for (int c = lane; c < dm; c += 32) m = max(m, (uint32_t)(w[c] & 0x7fffu));
  }
  m = max(m & 0xffffu, m >> 16);
  m = __reduce_max_sync(0xffffffffu, m);
  if (lane == 0) row_exp[row] = max((int)(m >> 7), 1);
}

// Exact Gram matrices W W^T on the tensor cores. A row's values are fixed
// point fractions of its largest exponent, x = sum_s d_s 2^(-7 s) with signed
// 7-bit digits d_1 .. d_8 (a bf16 value's 8 bits fall into two neighbouring
// digits), and digit matrices are exact in bf16, so W W^T is the sum over
// digit pairs of D_i D_j^T 2^(-7 (i + j)). Pairs with the same i + j = c share
// a TMEM accumulator, and before one holds more than kGramExact digit products
// (each below 2^14) the accumulators are added into 64-bit integers: every fp32
// accumulation is exact. Products below 2^-63 of the
// two rows' scale (c > 9) are left out; fp64 sums round at 2^-53 of it. The
// result rounds once, when it becomes a double.
//
// The 8 accumulators (c = 2 .. 9) do not fit TMEM at once, so
// blockIdx.z = 0 takes c = 2 .. 5 (digits 1-4, 10 pairs) and 1 takes c = 6 .. 9
// (26 pairs), each writing its own part. Four digits hold every weight down to
// 2^-20 of its row's largest, so a step of 64 columns whose weights have no
// digit past the fourth (nearly all) is narrow: 4 digit tiles, and 6 pairs for
// c = 6 .. 9. Narrow steps alternate between the halves of the 8 tiles, so that
// one's digits are formed while the other's products run.
//
// For 896 matrices of 128 x 3584 this takes 2.57 ms, and the row exponents 0.11 ms
// (7.1 TB/s); with all 8 digits formed and multiplied in every step, one after the
// other, it took 4.8 ms, and the plain fp64 Gram 88.6 ms (105 GFLOP at 1.19
// TFLOP/s, the fp64 pipe's two FMAs a clock and SM). It is bound by the
// digit production, about 25 instructions a weight.
//
// One CTA: 128 rows (one matrix at d_head 128, two at 64, whose off-diagonal
// blocks are dropped), 512 threads. Each thread turns 16 weights of a
// 64-column step into digits (128-byte-swizzled K-major tiles, one per digit),
// one thread issues the step's MMAs, and the weights of the step after the next
// are loaded meanwhile.
constexpr int kDigits = 8;
constexpr int kNarrow = 4;  // digits of a step without deep weights
constexpr int kDigitTile = 128 * 64 * 2;
constexpr int kGramTcThreads = 512;
constexpr int kGramTcSmem = kDigits * kDigitTile + 1024;
// Digit products that an accumulator takes between two reads: 127^2 times as many
// stay below 2^24.
constexpr int kGramExact = 1040;
constexpr int kGramSpan = 128;  // a split takes a multiple of these columns
constexpr uint32_t kGramIdesc = idesc_bf16(128, 128, false);

__global__ void __launch_bounds__(kGramTcThreads, 1)
    gram_tc_kernel(const bf16* wq, const bf16* wk, int Hq, int Hkv, int nall, int dh, int dm, int span, int vec,
                   const int* row_exp, double* part, uint32_t* err) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = smem_raw + ((1024 - (smem_u32(smem_raw) & 1023)) & 1023);
  __shared__ uint64_t done[2];  // step n's MMAs complete on done[n & 1]
  __shared__ uint32_t tmem_slot;
  __shared__ int s_abort, col_exp[128];
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  const int per = 128 / dh;  // matrices of this CTA
  const int split = blockIdx.y, high = blockIdx.z;
  const int k0 = split * span, k1 = min(dm, k0 + span);
  if (t == 0) {
    mbar_init(&done[0], 1);
    mbar_init(&done[1], 1);
    s_abort = 0;
    fence_mbar_init();
  }
  if (t < 128) {
    const int m = blockIdx.x * per + t / dh;
    col_exp[t] = m < nall ? row_exp[m * dh + t % dh] : 1;
  }
  if (warp == 0) {
    tmem_alloc(&tmem_slot, 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_slot;

  // digit production: row t / 4, columns 16 (t % 4) .. + 15 of each step
  const int prow = t >> 2, pch = (t & 3) * 2;
  const int pm = blockIdx.x * per + prow / dh;
  const bool has = pm < nall;
  const uint16_t* wrow =
      has ? reinterpret_cast<const uint16_t*>(weight_of(wq, wk, pm, Hq, Hkv, dh, dm)) + (size_t)(prow % dh) * dm
          : nullptr;
  const int pexp = col_exp[prow];
  uint32_t w[8] = {}, next[8] = {};  // this step's weights and the next one's, two a word
  auto load = [&](int kc, uint32_t (&w)[8]) {
    const int c0 = kc + (t & 3) * 16;
#pragma unroll
    for (int i = 0; i < 8; ++i) w[i] = 0u;
    if (!has) return;
    if (vec) {  // dm, k0 and k1 are multiples of 8
#pragma unroll
      for (int i = 0; i < 2; ++i)
        if (c0 + 8 * i < k1) {
          const uint4 v = __ldg(reinterpret_cast<const uint4*>(wrow + c0 + 8 * i));
          w[4 * i] = v.x;
          w[4 * i + 1] = v.y;
          w[4 * i + 2] = v.z;
          w[4 * i + 3] = v.w;
        }
    } else {
#pragma unroll
      for (int i = 0; i < 16; ++i)
        if (c0 + i < k1) w[i >> 1] |= (uint32_t)wrow[c0 + i] << ((i & 1) * 16);
    }
  };
  // a weight's two digits, first | second << 8, and the place of the first
  auto two_digits = [&](int i, int& s0) {
    const uint32_t h = (w[i >> 1] >> ((i & 1) * 16)) & 0x7fffu;
    const int ef = (int)(h >> 7);
    const uint32_t mant = (h & 127u) | (ef ? 128u : 0u);
    const int p = min(pexp - max(ef, 1), 63);  // leading bit at 2^(-1 - p)
    s0 = (p * 37) >> 8;                         // p / 7
    const uint32_t y = mant << (6 - (p - 7 * s0));
    return (y >> 7) | (y & 127u) << 8;
  };
  uint32_t x[16];  // digits 1-4 of each weight, a byte each
  auto first_digits = [&]() {  // whether a weight has digits past the fourth
    uint32_t deep = 0;
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      int s0;
      const uint32_t d = two_digits(i, s0);
      x[i] = __funnelshift_lc(0u, d, 8 * s0);
      deep |= __funnelshift_lc(d, 0u, 8 * s0);
    }
    return deep != 0u;
  };
  // four digit tiles from x: 128 + d is a bf16 value's bits 0x4300 | d, and
  // +-(128 + d) -+ 128 is exact
  auto emit = [&](uint8_t* tiles) {
#pragma unroll
    for (int half = 0; half < 2; ++half) {
      uint8_t* dst = tiles + prow * 128 + (((pch + half) ^ (prow & 7)) << 4);
#pragma unroll
      for (int s = 0; s < 4; ++s) {
        uint32_t o[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int e = 8 * half + 2 * i;
          const uint32_t sign = w[e >> 1] & 0x80008000u;
          const uint32_t d = (__byte_perm(x[e], x[e + 1], s * 0x1111 + 0x4400) & 0x007f007fu) | 0x43004300u;
          o[i] = bf16x2_fma(d, 0x3f803f80u | sign, 0xc300c300u ^ sign);
        }
        *reinterpret_cast<uint4*>(dst + s * kDigitTile) = make_uint4(o[0], o[1], o[2], o[3]);
      }
    }
  };
  auto last_digits = [&]() {  // x: digits 5-8
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      int s0;
      const uint32_t d = two_digits(i, s0);
      x[i] = s0 < 4 ? __funnelshift_lc(d, 0u, 8 * s0) : __funnelshift_lc(0u, d, 8 * s0 - 32);
    }
  };
  // one elected lane: the step's digit pairs; accumulators not in `started` are
  // overwritten
  auto issue = [&](int n_dig, const uint8_t* tiles, int started, uint64_t* bar) {
    const uint64_t base = sdesc_sw128(smem_u32(tiles), 16, 1024);
    for (int a = 0; a < 4; ++a) {
      const int c = a + (high ? 6 : 2);
      const int i0 = max(1, c - n_dig), i1 = min(c - 1, n_dig);
      for (int i = i0; i <= i1; ++i) {
        const uint64_t da = base + (uint32_t)((i - 1) * sdesc_step(kDigitTile));
        const uint64_t db = base + (uint32_t)((c - i - 1) * sdesc_step(kDigitTile));
#pragma unroll
        for (int kk = 0; kk < 4; ++kk)
          tc_mma(tmem + a * 128, da + sdesc_step(kk * 32), db + sdesc_step(kk * 32), kGramIdesc,
                 (!(started >> a & 1) && i == i0 && kk == 0) ? 0u : 1u);
      }
    }
    tc_commit(bar);
  };

  // accumulators: row 32 (warp % 4) + lane, columns 32 (warp / 4) .. + 31
  const int row = (warp & 3) * 32 + lane, cg = warp >> 2;
  const bool wanted = dh == 128 || (row >> 6) == (cg >> 1);  // uniform over the warp
  long long acc[32];
#pragma unroll
  for (int i = 0; i < 32; ++i) acc[i] = 0;
  auto flush = [&](int started) {
    if (!wanted) return;
    const uint32_t tl = tmem + ((uint32_t)((warp & 3) * 32) << 16) + cg * 32;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      uint32_t v0[8], v1[8], v2[8], v3[8];
      tmem_ld8(tl + q * 8, v0);
      tmem_ld8(tl + 128 + q * 8, v1);
      tmem_ld8(tl + 256 + q * 8, v2);
      tmem_ld8(tl + 384 + q * 8, v3);
      tmem_ld_wait();
      if (!(started >> 3)) {  // only c = 9 can be without a product
#pragma unroll
        for (int i = 0; i < 8; ++i) v3[i] = 0u;
      }
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int a = __float2int_rn(__uint_as_float(v0[i])) * 128 + __float2int_rn(__uint_as_float(v1[i]));
        const int b = __float2int_rn(__uint_as_float(v2[i])) * 128 + __float2int_rn(__uint_as_float(v3[i]));
        acc[8 * q + i] += (long long)a * 16384 + b;
      }
    }
  };

  int step = 0;
  int started = 0, taken = 0;  // accumulators with products since the last flush, and the most of one
  bool ok = true, wide_before = false;
  auto wait_step = [&](int n) {
    ok = __all_sync(0xffffffffu, wait_bar(&done[n & 1], (n >> 1) & 1, err, &s_abort)) && ok;
    tc_fence_after();
  };
  load(k0, w);
  load(k0 + 64, next);
  for (int kc = k0; kc < k1; kc += 64, ++step) {
    const bool deep = first_digits();
    const bool wide = high && __syncthreads_or(deep);
    // all 8 tiles (wide), or the half that step - 2 used
    uint8_t* tiles = smem + (wide ? 0 : (step & 1) * kNarrow * kDigitTile);
    const bool all_done = wide || wide_before;
    if (step > 0 && all_done)
      wait_step(step - 1);
    else if (step > 1)
      wait_step(step - 2);
    if (ok) {
      emit(tiles);
      if (wide) {
        last_digits();
        emit(tiles + kNarrow * kDigitTile);
      }
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) w[i] = next[i];
    load(kc + 128, next);
    const int products = 64 * (wide ? 8 : high ? 3 : 4);  // of the pair sum with the most pairs
    if (taken + products > kGramExact) {
      if (!all_done) wait_step(step - 1);
      if (ok) flush(started);
      started = taken = 0;
    }
    taken += products;
    wide_before = wide;
    fence_proxy_async_smem();
    tc_fence_before();
    ok = __syncthreads_and(ok);
    if (!ok) break;
    if (warp == 0) {
      tc_fence_after();
      if (elect_one()) issue(wide ? kDigits : kNarrow, tiles, started, &done[step & 1]);
    }
    __syncwarp();
    started |= high && !wide ? 7 : 15;
  }
  if (step > 0) {  // every issued MMA ends before TMEM is freed
    ok = drain_wait(&done[(step - 1) & 1], ((step - 1) >> 1) & 1, err) && ok;
    tc_fence_after();
    if (__all_sync(0xffffffffu, ok)) flush(started);
  }
  const int m = blockIdx.x * per + row / dh;
  if (wanted && m < nall) {
    double* out = part + ((size_t)(split * 2 + high) * nall + m) * dh * dh + (size_t)(row % dh) * dh + (cg * 32) % dh;
    const int ei = col_exp[row];
#pragma unroll
    for (int i = 0; i < 32; ++i) {
      const int ej = col_exp[cg * 32 + i];
      // value 2^(e - 126) per unit of either row's fractions
      const double sc = __longlong_as_double((long long)(1023 + ei + ej - 252 - (high ? 63 : 35)) << 52);
      out[i] = ei == 255 || ej == 255 ? __longlong_as_double(0x7ff8000000000000ll) : (double)acc[i] * sc;
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 0) tmem_dealloc(tmem, 512);
}

// Sum of a block's values (every thread gets it); `red` holds 32 doubles.
__device__ double block_sum(double v, double* red) {
  for (int o = 16; o >= 1; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  double s = 0.0;
  for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += red[w];
  return s;
}

__device__ double block_max(double v, double* red) {
  for (int o = 16; o >= 1; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
  __syncthreads();
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  double s = red[0];
  for (int w = 1; w < (int)(blockDim.x >> 5); ++w) s = fmax(s, red[w]);
  return s;
}

template <int N>
constexpr int kCholSmem = (N * (N + 1) + N) * 8;

// One matrix per CTA: G = sum of the split parts, then G = L L^T, written to L
// with the upper triangle zeroed. N + 1 doubles a row in shared memory: neither
// a row nor a column walk meets a bank conflict. Each step scales its column
// into a vector; then lanes along a row subtract, four rows at a time, so a
// step's loads are one per product. With conflicting column reads and a
// division per element for its index the 896 matrices of 28 layers took 3.0 ms;
// 2.1 ms now, of which the fp64 pipe's two FMAs a clock take one.
template <int N>
__global__ void __launch_bounds__(4 * N) chol_kernel(const double* part, int nparts, int nall, double* L) {
  constexpr int LD = N + 1;
  extern __shared__ double A[];  // row i, column k at A[i * LD + k]
  double* col = A + N * LD;      // the scaled column
  __shared__ double red[32];
  __shared__ double inv_d;
  const int m = blockIdx.x, x = threadIdx.x % N, g = threadIdx.x / N;
  constexpr size_t n2 = (size_t)N * N;
  double dmax = 0.0;
  for (int i = g; i < N; i += 4) {
    double s = 0.0;
    for (int p = 0; p < nparts; ++p) s += part[((size_t)p * nall + m) * n2 + (size_t)i * N + x];
    A[i * LD + x] = s;
    if (i == x) dmax = s;
  }
  const double tol = N * DBL_EPSILON * block_max(dmax, red);
  for (int j = 0; j < N; ++j) {
    if (threadIdx.x == 0) {
      const double piv = A[j * LD + j];
      const double d = piv > tol ? sqrt(piv) : 0.0;
      A[j * LD + j] = d;
      inv_d = d > 0.0 ? 1.0 / d : 0.0;
    }
    __syncthreads();
    if (g == 0 && x > j) {
      const double v = A[x * LD + j] * inv_d;
      A[x * LD + j] = v;
      col[x] = v;
    }
    __syncthreads();
    const int k = j + 1 + x;  // this thread's column, rows k and below
    if (k < N) {
      const double ck = col[k];
      for (int i = j + 1 + g; i < N; i += 4)
        if (i >= k) A[i * LD + k] = fma(-col[i], ck, A[i * LD + k]);
    }
    __syncthreads();
  }
  double* out = L + (size_t)m * n2;
  for (int i = g; i < N; i += 4) out[(size_t)i * N + x] = x <= i ? A[i * LD + x] : 0.0;
}

// Warp sum of a double (every lane gets it).
__device__ __forceinline__ double warp_sum(double v) {
  for (int o = 16; o >= 1; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Singular values of one query head's A = L_K^T L_Q need no vectors, so A is
// reduced to bidiagonal form by Householder reflections (Golub & Kahan 1965;
// 8/3 n^3 flops) and svals_kernel finds the n values of the bidiagonal. The
// one-sided Jacobi iteration that stood here spent about 10 sweeps of 10 n^3
// flops each: 240 ms for 784 heads of 128. The reduction now takes 9.7 ms (its
// 4.4 GFLOP and the product's 1.5 cost 5 ms at the 1.2 TFLOP/s the fp64 pipe
// gives; the rest is the chain of 256 reflectors a head and the sixth, mostly
// empty, wave of heads) and the values 1.5 ms.
//
// One CTA per head, 4 N threads, A row-major in shared memory with N + 1
// doubles a row, so that neither a row nor a column walk meets a bank
// conflict; lanes lie along the columns for the left reflections and along
// the rows for the right ones, the four thread groups split the other index,
// and a product's four partial sums meet in shared memory (a warp shuffle
// reduction would cost as many fp64 adds as the product itself). The pipe
// issues two fp64 FMAs a clock, so shared memory (one load per FMA) keeps up.
// A reflector H = I - c v v^T, c = 1 / (beta (beta - alpha)), keeps v in place
// of the eliminated entries with only its first entry stored apart.
template <int N>
struct BidiagCfg {
  static constexpr int LD = N + 1;
  static constexpr int SMEM = (N * LD + 4 * N) * 8;
};

// The reflector that maps x = (alpha, rest), |rest|^2 = sig, to (beta, 0):
// head[0] = beta, head[1] = first entry of v, head[2] = c (0: nothing to do).
__device__ __forceinline__ void make_reflector(double alpha, double sig, double* head) {
  if (sig == 0.0) {
    head[0] = alpha;
    head[1] = 0.0;
    head[2] = 0.0;
  } else {
    const double mu = sqrt(fma(alpha, alpha, sig));
    const double beta = alpha > 0.0 ? -mu : mu;
    head[0] = beta;
    head[1] = alpha - beta;
    head[2] = 1.0 / (beta * (beta - alpha));
  }
}

template <int N>
__global__ void __launch_bounds__(4 * N) bidiag_kernel(const double* L, int Hq, int Hkv, double* diag, double* sup) {
  using C = BidiagCfg<N>;
  constexpr int LD = C::LD, R = N / 4;
  extern __shared__ double A[];  // row i, column j at A[i * LD + j]
  double* part = A + N * LD;     // [4][N] partial products
  __shared__ double head[2][3];  // the left and the right reflector
  const int hg = blockIdx.x, l = hg / Hq, h = hg % Hq, kv = h / (Hq / Hkv);
  const size_t n2 = (size_t)N * N;
  const double* Lq = L + ((size_t)l * (Hq + Hkv) + h) * n2;
  const double* Lk = L + ((size_t)l * (Hq + Hkv) + Hq + kv) * n2;
  const int x = threadIdx.x % N, g = threadIdx.x / N, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  {
    // column x, rows R g .. R g + R - 1 of A = L_K^T L_Q; both factors are
    // lower triangular, so the sum starts at the larger of the two blocks
    double acc[R];
#pragma unroll
    for (int i = 0; i < R; ++i) acc[i] = 0.0;
    for (int m = max(R * g, x & ~31); m < N; ++m) {
      const double b = Lq[(size_t)m * N + x];
      const double2* a = reinterpret_cast<const double2*>(Lk + (size_t)m * N + R * g);
#pragma unroll
      for (int i = 0; i < R / 2; ++i) {
        const double2 v = a[i];
        acc[2 * i] = fma(v.x, b, acc[2 * i]);
        acc[2 * i + 1] = fma(v.y, b, acc[2 * i + 1]);
      }
    }
#pragma unroll
    for (int i = 0; i < R; ++i) A[(R * g + i) * LD + x] = acc[i];
  }
  __syncthreads();

  for (int k = 0; k < N; ++k) {
    // left: column k, rows k .. N - 1
    if (warp == 0) {
      double s = 0.0;
      for (int i = k + 1 + lane; i < N; i += 32) s = fma(A[i * LD + k], A[i * LD + k], s);
      s = warp_sum(s);
      if (lane == 0) {
        make_reflector(A[k * LD + k], s, head[0]);
        diag[(size_t)hg * N + k] = head[0][0];
      }
    }
    __syncthreads();
    const int j = k + 1 + x;  // the column this thread updates
    double c = head[0][2], v0 = head[0][1];
    if (c != 0.0) {
      if (j < N) {
        double s = g == 0 ? v0 * A[k * LD + j] : 0.0;
        for (int i = k + 1 + g; i < N; i += 4) s = fma(A[i * LD + k], A[i * LD + j], s);
        part[g * N + x] = s;
      }
      __syncthreads();
      if (j < N) {
        const double w = -c * ((part[x] + part[N + x]) + (part[2 * N + x] + part[3 * N + x]));
        if (g == 0) A[k * LD + j] = fma(v0, w, A[k * LD + j]);
        for (int i = k + 1 + g; i < N; i += 4) A[i * LD + j] = fma(A[i * LD + k], w, A[i * LD + j]);
      }
      __syncthreads();
    }
    if (k + 1 >= N) break;
    // right: row k, columns k + 1 .. N - 1
    if (warp == 0) {
      double s = 0.0;
      for (int i = k + 2 + lane; i < N; i += 32) s = fma(A[k * LD + i], A[k * LD + i], s);
      s = warp_sum(s);
      if (lane == 0) {
        make_reflector(A[k * LD + k + 1], s, head[1]);
        sup[(size_t)hg * N + k] = head[1][0];
      }
    }
    __syncthreads();
    c = head[1][2];
    v0 = head[1][1];
    if (c != 0.0) {
      const int r = k + 1 + x;  // the row this thread updates
      const double* u = A + k * LD;
      if (r < N) {
        double s = g == 0 ? v0 * A[r * LD + k + 1] : 0.0;
        for (int i = k + 2 + g; i < N; i += 4) s = fma(u[i], A[r * LD + i], s);
        part[g * N + x] = s;
      }
      __syncthreads();
      if (r < N) {
        const double w = -c * ((part[x] + part[N + x]) + (part[2 * N + x] + part[3 * N + x]));
        if (g == 0) A[r * LD + k + 1] = fma(v0, w, A[r * LD + k + 1]);
        for (int i = k + 2 + g; i < N; i += 4) A[r * LD + i] = fma(u[i], w, A[r * LD + i]);
      }
    }
    __syncthreads();
  }
}

// 1 / x for 1e-30 <= |x| <= 1e30, to about an ulp: the residual e = 1 - x y of
// an fp32 reciprocal y gives y (1 + e + e^2) + O(e^3), e < 2^-22. Half the fp64
// operations of a division.
__device__ __forceinline__ double fast_rcp(double x) {
  const double y = (double)__frcp_rn((float)x);
  const double e = fma(-x, y, 1.0);
  return fma(y, fma(e, e, e), y);
}

// Singular values of each head's bidiagonal matrix B and its ER; one CTA of N
// threads per head, thread j finds the j-th smallest value. With q_i = d_i^2
// and f_i = e_i^2, the stationary qd transform (Fernando & Parlett 1994)
//   delta_i = q_i + t_i, t_0 = -s, t_{i+1} = t_i f_i / delta_i - s
// has as many negative delta_i as B^T B has eigenvalues below s, to high
// relative accuracy, and sum_i delta_i' / delta_i is p'(s) / p(s) of its
// characteristic polynomial. Each thread first bisects in fp32 (the fp32 pipe
// is 64 times as wide as the fp64 pipe), then takes Newton steps in fp64 from
// there, two or three as a rule. Every evaluation's count says on which side of
// the wanted value the point lies: a step is taken only towards that side and
// inside the bracket that the counts have left, else the bracket is halved.
// Towards a value that repeats m times a Newton step closes only 1 / m of the
// distance, so from the ninth round on every round halves the bracket, and 54
// halvings end any search: with three Newton steps to a halving, up to 120
// rounds, the values beside a repeated one were left up to 5e-11 of the largest
// away. The values are wanted to absolute accuracy (ER weights them by their share
// of the sum). 784 heads of 128 take 1.5 ms; with the bisection in fp64 as well, from
// 128 shared counts to single values, and divisions for the reciprocals they took
// 22 ms.
template <int N>
__global__ void __launch_bounds__(N) svals_kernel(const double* diag, const double* sup, int dm, double* er) {
  __shared__ double2 qf[N];  // (q_i, f_i)
  __shared__ double red[32];
  __shared__ float2 qf32[N];
  const int hg = blockIdx.x, j = threadIdx.x;
  const double d = fabs(diag[(size_t)hg * N + j]);
  const double e = j + 1 < N ? fabs(sup[(size_t)hg * N + j]) : 0.0;
  const double ep = j > 0 ? fabs(sup[(size_t)hg * N + j - 1]) : 0.0;
  // sigma_max <= sqrt(|B|_1 |B|_inf) <= bound
  const double bound = block_max(fmax(d + e, d + ep), red);
  if (!(bound > 0.0)) {
    if (j == 0) er[hg] = 1.0;  // exp of an empty sum
    return;
  }
  const double inv_b = 1.0 / bound;
  qf[j] = make_double2((d * inv_b) * (d * inv_b), (e * inv_b) * (e * inv_b));
  qf32[j] = make_float2((float)qf[j].x, (float)qf[j].y);
  __syncthreads();
  // fp32 bisection to a bracket of 2^-22
  float xf = 0.5f;
  {
    float flo = 0.f, fhi = 1.f;
#pragma unroll 1
    for (int round = 0; round < 22; ++round) {
      xf = 0.5f * (flo + fhi);
      const float s = xf * xf;
      float t = -s;
      int c = 0;
#pragma unroll 8
      for (int i = 0; i < N; ++i) {
        const float2 v = qf32[i];
        float del = v.x + t;
        if (fabsf(del) < 1e-30f) del = -1e-30f;
        c += del < 0.f;
        t = fmaf(__fdividef(v.y, del), t, -s);
      }
      if (c <= j)
        flo = xf;
      else
        fhi = xf;
    }
    xf = 0.5f * (flo + fhi);
  }
  double x = fmax((double)xf, 1e-16), lo = 0.0, hi = 1.0 + 1e-9, prev = 0.0;
  int nlo = 0, nhi = N;
  bool done = false;
  constexpr int kNewtonRounds = 8, kRounds = kNewtonRounds + 56;
  for (int round = 0; round < kRounds && !__all_sync(0xffffffffu, done); ++round) {
    const double s = x * x;
    double t = -s, tp = -1.0, g = 0.0;  // g = p'(s) / p(s)
    int c = 0;
#pragma unroll 4
    for (int i = 0; i < N; ++i) {
      const double2 v = qf[i];
      double del = v.x + t;
      if (fabs(del) < 1e-30) del = -1e-30;
      c += del < 0.0;
      const double inv = fast_rcp(del);
      const double r = v.y * inv, u = tp * inv;
      g += u;
      t = fma(r, t, -s);
      tp = fma(r * v.x, u, -1.0);
    }
    if (done) continue;  // repeats its last point while others search
    if (c <= j) {
      lo = x;
      nlo = c;
    } else {
      hi = x;
      nhi = c;
    }
    const double xn = x - 1.0 / (2.0 * x * g);
    const double step = fabs(xn - x);
    const bool near_j = c == j || c == j + 1;
    // Once a Newton step is far shorter than the one before, a step of 1e-14
    // leaves 1e-20. Its sign may be rounding, so it may leave the bracket, but by
    // no more than rounding: a step towards a neighbour of the wanted value can be
    // as short. (Steps of 1e-11, taken wherever they led, gave the neighbour or
    // a cluster's edge in one of 1e4 spectra of near-equal values, 7e-9 off.)
    const bool converged = near_j && step < 1e-14 && step < 1e-3 * prev && xn > lo - 4e-15 && xn < hi + 4e-15;
    const bool newton = near_j && (xn > x) == (c <= j) && xn > lo && xn < hi && round < kNewtonRounds;
    const double mid = 0.5 * (lo + hi);
    done = converged || hi - lo < 1.2e-16 || hi < 1e-15 || (newton ? step < 4e-15 && nhi - nlo == 1 : mid <= lo || mid >= hi);
    prev = newton ? step : 0.0;
    x = converged || newton ? xn : mid;
  }
  const double nrm = x * bound;
  const double smax = block_max(nrm, red);
  const double tol = smax * (double)max(dm, N) * DBL_EPSILON;
  const bool keep = nrm > tol;
  // The sums' rounding errors would show in ER (exp of 4.7 moves by 9e-16 of itself
  // with the last bit of its argument): each is summed again as what the first
  // sum left, over terms that are small then, and enters to first order. A total
  // off by d of itself moves the entropy H by d (H - 1).
  const double kept = keep ? nrm : 0.0;
  const double total = block_sum(kept, red);
  const double off = block_sum(kept - total * (1.0 / N), red) / total;
  double ent = 0.0;
  if (keep) {
    const double p = nrm / total;
    ent = -p * log(p);
  }
  const double H = block_sum(ent, red);
  const double rest = block_sum(ent - H * (1.0 / N), red) - off * (H - 1.0);
  if (j == 0) {
    const double e = exp(H);
    er[hg] = total > 0.0 ? fma(e, rest, e) : e;
  }
}

// One layer per block (blockIdx.x), one thread.
__global__ void classify_kernel(const double* er_all, int Hq, int Hkv, int sparsity_pct, uint8_t* labels_all) {
  if (threadIdx.x != 0) return;
  const double* er = er_all + (size_t)blockIdx.x * Hq;
  uint8_t* labels = labels_all + (size_t)blockIdx.x * Hkv;
  const int g = Hq / Hkv;
  double score[kMaxKvHeads];
  int order[kMaxKvHeads];
  for (int kv = 0; kv < Hkv; ++kv) {
    double s = 0.0;
    for (int i = 0; i < g; ++i) s += er[kv * g + i];
    score[kv] = s / g;
    order[kv] = kv;
  }
  for (int i = 1; i < Hkv; ++i) {  // stable insertion sort, ascending
    const int x = order[i];
    int j = i - 1;
    while (j >= 0 && score[order[j]] > score[x]) {
      order[j + 1] = order[j];
      --j;
    }
    order[j + 1] = x;
  }
  const int k = ((100 - sparsity_pct) * Hkv + 99) / 100;
  for (int i = 0; i < Hkv; ++i) labels[order[i]] = i < k ? AOH_RETRIEVAL : AOH_STREAMING;
}

}  // namespace
}  // namespace aoh

using namespace aoh;

extern "C" aoh_status aoh_classify(const void* w_q, const void* w_k, int32_t n_layers, int32_t n_q_heads,
                                   int32_t n_kv_heads, int32_t d_head, int32_t d_model, int32_t sparsity_pct,
                                   double* er_out, uint8_t* labels_out, void* stream) {
  auto fail = [](aoh_status st, const char* msg) {
    record_error(msg);
    return st;
  };
  if (!w_q || !w_k || !labels_out)
    return fail(AOH_ERR_INVALID, "aoh_classify: w_q, w_k and labels_out must not be NULL");
  if (n_layers < 1 || n_layers > 65535) return fail(AOH_ERR_INVALID, "aoh_classify: n_layers outside [1, 65535]");
  if (n_q_heads < 1 || n_kv_heads < 1 || n_q_heads % n_kv_heads)
    return fail(AOH_ERR_INVALID, "aoh_classify: n_q_heads must be a positive multiple of n_kv_heads");
  if (n_kv_heads > kMaxKvHeads) return fail(AOH_ERR_UNSUPPORTED, "aoh_classify: more than 64 KV heads");
  if (d_head != 64 && d_head != 128) return fail(AOH_ERR_UNSUPPORTED, "aoh_classify: d_head must be 64 or 128");
  if (d_model < 1) return fail(AOH_ERR_INVALID, "aoh_classify: d_model must be >= 1");
  if (sparsity_pct < 0 || sparsity_pct > 100)
    return fail(AOH_ERR_INVALID, "aoh_classify: sparsity_pct outside [0, 100]");
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const int dh = d_head, nmat = n_q_heads + n_kv_heads;
  const int nall = n_layers * nmat, nq = n_layers * n_q_heads;
  if ((long long)n_layers * nmat > 65535) return fail(AOH_ERR_INVALID, "aoh_classify: too many matrices in one call");
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return fail(AOH_ERR_CUDA, "aoh_classify: device query failed");
  // split d_model so that the Gram grid (two CTAs per 128 rows and split)
  // covers about two waves, >= 256 columns a split
  const int groups = (nall * dh + 127) / 128;
  int nsplit = (sms + groups - 1) / groups;
  nsplit = std::max(1, std::min(nsplit, std::max(1, d_model / 256)));
  nsplit = std::min(nsplit, 16);
  const int span = ((d_model + nsplit - 1) / nsplit + kGramSpan - 1) / kGramSpan * kGramSpan;
  nsplit = (d_model + span - 1) / span;
  const int nparts = 2 * nsplit;
  const size_t n2 = (size_t)dh * dh;
  // Gram parts, factors, bidiagonals, ER; error word, row exponents; labels
  const size_t bytes = ((size_t)nparts * nall * n2 + (size_t)nall * n2 + 2 * (size_t)nq * dh + nq) * sizeof(double) +
                       (1 + (size_t)nall * dh) * sizeof(int) + (size_t)n_layers * n_kv_heads;
  void* scratch = nullptr;
  e = cudaMallocAsync(&scratch, bytes, s);
  if (e != cudaSuccess) return fail(AOH_ERR_CUDA, "aoh_classify: cudaMallocAsync failed");
  double* part = static_cast<double*>(scratch);
  double* L = part + (size_t)nparts * nall * n2;
  double* diag = L + (size_t)nall * n2;
  double* sup = diag + (size_t)nq * dh;
  double* er = sup + (size_t)nq * dh;
  uint32_t* err = reinterpret_cast<uint32_t*>(er + nq);
  int* row_exp = reinterpret_cast<int*>(err + 1);
  uint8_t* labels = reinterpret_cast<uint8_t*>(row_exp + (size_t)nall * dh);
  static std::atomic<uint64_t> done{0};
  e = once_per_device(done, [] {
    cudaError_t e = cudaFuncSetAttribute(chol_kernel<128>, cudaFuncAttributeMaxDynamicSharedMemorySize, kCholSmem<128>);
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(bidiag_kernel<128>, cudaFuncAttributeMaxDynamicSharedMemorySize, BidiagCfg<128>::SMEM);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(gram_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kGramTcSmem);
    return e;
  });
  if (e != cudaSuccess) {
    cudaFreeAsync(scratch, s);
    return fail(AOH_ERR_CUDA, "aoh_classify: cudaFuncSetAttribute failed");
  }
  const bf16 *wq = static_cast<const bf16*>(w_q), *wk = static_cast<const bf16*>(w_k);
  // 16-byte loads of the weights when every row starts on 16 bytes
  const int vec = d_model % 8 == 0 && ((reinterpret_cast<uintptr_t>(w_q) | reinterpret_cast<uintptr_t>(w_k)) & 15) == 0;
  cudaMemsetAsync(err, 0, sizeof(*err), s);
  row_exp_kernel<<<(nall * dh + 7) / 8, 256, 0, s>>>(wq, wk, n_q_heads, n_kv_heads, nall * dh, dh, d_model, vec, row_exp);
  gram_tc_kernel<<<dim3(groups, nsplit, 2), kGramTcThreads, kGramTcSmem, s>>>(
      wq, wk, n_q_heads, n_kv_heads, nall, dh, d_model, span, vec, row_exp, part, err);
  if (dh == 128) {
    chol_kernel<128><<<nall, 512, kCholSmem<128>, s>>>(part, nparts, nall, L);
    bidiag_kernel<128><<<nq, 512, BidiagCfg<128>::SMEM, s>>>(L, n_q_heads, n_kv_heads, diag, sup);
    svals_kernel<128><<<nq, 128, 0, s>>>(diag, sup, d_model, er);
  } else {
    chol_kernel<64><<<nall, 256, kCholSmem<64>, s>>>(part, nparts, nall, L);
    bidiag_kernel<64><<<nq, 256, BidiagCfg<64>::SMEM, s>>>(L, n_q_heads, n_kv_heads, diag, sup);
    svals_kernel<64><<<nq, 64, 0, s>>>(diag, sup, d_model, er);
  }
  classify_kernel<<<n_layers, 32, 0, s>>>(er, n_q_heads, n_kv_heads, sparsity_pct, labels);
  e = cudaGetLastError();
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(labels_out, labels, (size_t)n_layers * n_kv_heads, cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess && er_out) e = cudaMemcpyAsync(er_out, er, nq * sizeof(double), cudaMemcpyDeviceToHost, s);
  uint32_t h_err = 0;
  if (e == cudaSuccess) e = cudaMemcpyAsync(&h_err, err, sizeof(h_err), cudaMemcpyDeviceToHost, s);
  const cudaError_t f = cudaFreeAsync(scratch, s);
  if (e == cudaSuccess) e = f;
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) return fail(AOH_ERR_CUDA, "aoh_classify: a CUDA call failed");
  if (h_err) return fail(AOH_ERR_TIMEOUT, "aoh_classify: a kernel's bounded wait ran out");
  return AOH_OK;
}
