// Host runtime behind include/aoh.h: argument validation, cache layout,
// split-KV scheduling and kernel launches on the caller's stream.
#include <math.h>
#include <stdarg.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

#include <algorithm>
#include <functional>
#include <string>
#include <vector>

#include "../../include/aoh.h"
#include "internal.h"

using namespace aoh;

namespace {

thread_local std::string g_last_error;

aoh_status fail(aoh_status st, const char* fmt, ...) {
  char buf[512];
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(buf, sizeof(buf), fmt, ap);
  va_end(ap);
  g_last_error = buf;
  return st;
}

aoh_status cuda_fail(cudaError_t e, const char* what) {
  return fail(AOH_ERR_CUDA, "%s: %s", what, cudaGetErrorString(e));
}

bool aligned(const void* p, size_t a) { return (reinterpret_cast<uintptr_t>(p) % a) == 0; }

// Validates cfg + labels; fills n_r / n_s. Returns AOH_OK or an error.
aoh_status check_config(const aoh_config* cfg, const uint8_t* labels, int* n_r, int* n_s) {
  if (!cfg) return fail(AOH_ERR_INVALID, "cfg is NULL");
  if (!labels) return fail(AOH_ERR_INVALID, "head_labels is NULL");
  const aoh_config& c = *cfg;
  if (c.batch < 1 || c.n_q_heads < 1 || c.n_kv_heads < 1 || c.max_seq < 1)
    return fail(AOH_ERR_INVALID, "batch, n_q_heads, n_kv_heads and max_seq must be >= 1");
  if (c.n_kv_heads > kMaxKvHeads) return fail(AOH_ERR_UNSUPPORTED, "n_kv_heads > %d", kMaxKvHeads);
  if (c.n_q_heads % c.n_kv_heads) return fail(AOH_ERR_INVALID, "n_q_heads must be a multiple of n_kv_heads");
  if (c.d_head != 64 && c.d_head != 128) return fail(AOH_ERR_UNSUPPORTED, "d_head must be 64 or 128");
  if (c.sink < 0 || c.window < 1) return fail(AOH_ERR_INVALID, "need sink >= 0 and window >= 1");
  if (c.chunk < 0) return fail(AOH_ERR_INVALID, "chunk must be >= 0");
  int r = 0, s = 0;
  for (int h = 0; h < c.n_kv_heads; ++h) {
    if (labels[h] == AOH_RETRIEVAL)
      ++r;
    else if (labels[h] == AOH_STREAMING)
      ++s;
    else
      return fail(AOH_ERR_INVALID, "head_labels[%d] = %d is neither retrieval (0) nor streaming (1)", h,
                  (int)labels[h]);
  }
  *n_r = r;
  *n_s = s;
  return AOH_OK;
}

// Prefill work: items of two 128-row query tiles, heaviest first so the
// hardware block scheduler fills the machine longest-processing-time first. An
// item is one query tile of two heads of a group, or, for the last head of an
// odd group, two consecutive tiles of that head. Two heads see the same keys;
// two tiles visit the union of their KV tiles, so that each pair of tiles has one
// KV tile that the first does not see, and a sequence's last pair may lack the
// second: 8 ragged sequences of up to 2,999 tokens, 32/8 heads of 128 of which
// half stream (S = 64, W = 512), 298 -> 277 us; 32K tokens of 28/4 streaming heads
// (S = 128, W = 1024) 517 -> 480, 32K with half of them retrieval 2504 -> 2468.
// The cost, the number of KV tiles visited, is the same for all items of a kind,
// so (b, index, kind) entries are sorted and then expanded. *costs receives each
// item's cost.
std::vector<uint64_t> prefill_schedule(const CacheGeom& g, const std::vector<int32_t>& base,
                                       const std::vector<int32_t>& lens, std::vector<int>* costs) {
  constexpr int BM = 128, BN = 128;
  struct Entry {
    int cost, b, index;
    bool streaming, two_heads;
  };
  std::vector<Entry> entries;
  for (int b = 0; b < g.B; ++b) {
    const int Lb = base[b];
    const int S_rel = g.S - Lb;
    for (int streaming = 0; streaming < 2; ++streaming) {
      if ((streaming ? g.n_s : g.n_r) == 0) continue;
      const int n_c = Lb == 0 ? 0 : ((streaming ? std::min(Lb, g.S + g.W) : Lb) + BN - 1) / BN;
      for (int two_heads = 0; two_heads < 2; ++two_heads) {
        if ((two_heads ? g.G / 2 : g.G % 2) == 0) continue;
        const int rows = two_heads ? BM : 2 * BM;
        for (int q0 = 0; q0 < lens[b]; q0 += rows) {
          const int q_end = std::min(q0 + rows, (int)lens[b]);
          int n;
          if (!streaming) {
            n = (q_end + BN - 1) / BN;
          } else {
            const int a_end = (std::min(std::max(S_rel, 0), q_end) + BN - 1) / BN;
            const int c_begin = std::max(a_end, std::max(0, g.wstart(q0)) / BN);
            const int c_end = std::max(c_begin, (q_end + BN - 1) / BN);
            n = a_end + (c_end - c_begin);
          }
          entries.push_back({n_c + n, b, q0 / rows, streaming != 0, two_heads != 0});
        }
      }
    }
  }
  std::stable_sort(entries.begin(), entries.end(), [](const Entry& x, const Entry& y) { return x.cost > y.cost; });
  std::vector<uint64_t> items;
  const size_t most = entries.size() * (size_t)(g.Hq / 2 + g.Hkv);
  items.reserve(most);
  costs->reserve(most);
  for (const Entry& e : entries)
    for (int i = 0; i < (e.streaming ? g.n_s : g.n_r); ++i) {
      const int kvh = e.streaming ? g.s_head[i] : g.r_head[i];
      const int first = e.two_heads ? 0 : g.G - 1, step = e.two_heads ? 2 : 1;
      for (int h = first; h + step <= g.G; h += step) {
        items.push_back(prefill_item(e.b, kvh * g.G + h, e.index) | (e.two_heads ? kPrefillTwoHeads : 0));
        costs->push_back(e.cost);
      }
    }
  return items;
}

// The work of clusters of two CTAs, two entries a cluster: two items, or one item
// twice, with kPrefillHalf, that its CTAs share (kPrefillNone fills the last
// cluster). Nothing when one CTA an item is as good.
//
// When every item's cluster runs at once, the call lasts as long as its longest
// item, and sharing all halves that. Measured (8 heads of 128, one sequence, us of
// a call without / with): 512 rows (4 tiles) 17 / 18, 640 19 / 20, 1024 22 / 21, 2048
// 33 / 26; heads of 64: 512 16 / 16, 1024 20 / 18, 2048 30 / 22.
//
// In a few waves, as in a chunk after a long prefix whose heavy items all read it,
// a last wave of heavy items that leaves many SMs idle is shared, while the
// lighter items behind it are not. k + 1 of the first k * num_sms + 1 items meet
// on one SM; where that ends a tenth later than the work spread evenly, the ends
// of longest-first schedules decide, in visited tiles, with 4 tiles' time added
// to an item and 8 to a half: nothing shared, or half a wave or a whole one from
// item k * num_sms on (from the even one below, with an odd count of SMs). Past four items an SM the last wave matters little. 28
// heads of 128, half of them streaming (S = 128, W = 2048), us of a call without /
// with: 4096 rows after 16K tokens 388 / 388 (not shared), 20K 471 / 461, 24K 555 /
// 526, 28K 638 / 585; 1024 rows after 24K 272 / 151.
std::vector<uint64_t> prefill_pairs(const std::vector<uint64_t>& items, const std::vector<int>& costs, int num_sms) {
  const int n = (int)items.size(), slots = num_sms / 2;
  int first = 0, last = 0;  // items [first, last) are shared
  if (n <= slots) {
    if (n > 0 && costs[0] >= 7) last = n;
  } else if (n <= std::min(4 * num_sms, kPrefillSplitMost)) {
    long long work = 0, meet = 0;
    for (int c : costs) work += c + 4;
    for (int a = 0; a < n; a += num_sms)
      if ((a / num_sms + 1) * (long long)(costs[a] + 4) > meet) {
        meet = (a / num_sms + 1) * (long long)(costs[a] + 4);
        first = a;
      }
    first &= ~1;  // the halves of an item are entries 2 i and 2 i + 1 at any count of SMs
    if (meet * num_sms * 10 > work * 11) {
      std::vector<int> free_at;  // a min-heap
      auto end_of = [&](int count, int shared_end) {
        free_at.assign(count, 0);
        int end = 0;
        for (int i = 0; i < n;) {
          const bool half = i >= first && i < shared_end;
          std::pop_heap(free_at.begin(), free_at.end(), std::greater<int>());
          end = std::max(end, free_at.back() += half ? (costs[i] + 1) / 2 + 8 : costs[i] + 4);
          std::push_heap(free_at.begin(), free_at.end(), std::greater<int>());
          i += count == num_sms || half ? 1 : 2;
        }
        return end;
      };
      int best = end_of(num_sms, 0);
      for (int window = slots; window <= 2 * slots; window += slots) {
        const int end = end_of(slots, first + window);
        if (end < best) {
          best = end;
          last = std::min(first + window, n);
        }
      }
    }
  }
  std::vector<uint64_t> pairs;
  if (last == 0) return pairs;
  pairs.reserve(n + last - first + 2);
  for (int i = 0; i < n; ++i) {
    const bool half = i >= first && i < last;
    if (half) pairs.push_back(items[i] | kPrefillHalf);
    pairs.push_back(items[i] | (half ? kPrefillHalf : 0));
  }
  if (pairs.size() & 1) pairs.push_back(kPrefillNone);
  return pairs;
}

// Whether one CTA an SM goes through all items in one pipeline instead of a CTA an
// item: many short items, whose starts and ends it overlaps. It deals them out
// beforehand, which needs several for an SM to even out, and its loop over KV tiles
// is a few percent slower. Measured, us of a call with a CTA an item / so (32/8 heads
// of 128, half streaming, S = 64, W = 512; items an SM, tiles an item): 8 x 512 (3.4,
// 2.5) 41 / 38, 16 x 512 (6.7, 2.5) 78 / 62, 8 x 1024 (6.7, 4.3) 94 / 79, 2 x 2048
// (3.4, 6.8) 60 / 62, 8 x 2048 (13.5, 6.8) 220 / 191, 1 x 4096 (3.4, 11) 80 / 87, 2 x 4096
// (6.7, 11) 154 / 146, 1 x 8192 (6.7, 19) 224 / 238, 2 x 8192 (13.5, 19) 439 / 433; 4 x 512
// (1.7, 2.5) 24 / 25; 32K tokens of 28/4 heads (24, 73) 2469 / 2609.
bool prefill_is_short(const std::vector<int>& costs, int num_sms) {
  const long long n = (long long)costs.size();
  long long tiles = 0;
  for (int c : costs) tiles += c;
  return n >= 3 * num_sms && tiles <= 20 * n && tiles * num_sms * 10 <= 19 * n * n;
}

size_t bytes_for(const aoh_config& c, int n_r, int n_s) {
  const size_t tokens = (size_t)n_r * c.max_seq + (size_t)n_s * (size_t)(c.sink + c.window);
  return (size_t)c.batch * tokens * c.d_head * 2 * 2;
}

}  // namespace

void aoh::record_error(const char* msg) { g_last_error = msg; }

struct aoh_cache {
  DecodeArgs maps;  // the decode step's tensor maps (built once: the buffer does not move)
  aoh_config cfg;
  CacheGeom geom;
  std::vector<uint8_t> labels;
  void* kv = nullptr;
  size_t kv_bytes = 0;
  std::vector<int32_t> lens;  // host mirror of the device lengths
  // a call of this handle was captured into a graph, whose replays move the device
  // lengths alone: from then on the mirror does not place prefill chunks
  bool captured = false;
  int device = 0;
  int num_sms = 0;
  // device metadata (one allocation)
  void* meta = nullptr;
  int32_t* d_lens = nullptr;
  int32_t* d_chunk = nullptr;  // rows of the current prefill chunk
  uint32_t* d_counters = nullptr;
  uint32_t* d_gcounters = nullptr;
  uint32_t* d_done = nullptr;
  uint32_t* d_err = nullptr;
  float* d_partials = nullptr;
  // prefill work list (device), grown on demand
  uint64_t* d_work = nullptr;
  size_t work_cap = 0;
  // H2Share anchor workspace (scores, head states, importance overflow),
  // allocated on first use
  float* d_h2 = nullptr;
};

namespace {

// Grow the prefill work list to at least n items (cudaMalloc, which
// synchronises the device).
cudaError_t reserve_work(aoh_cache* h, size_t n) {
  if (n <= h->work_cap) return cudaSuccess;
  if (h->d_work) cudaFree(h->d_work);
  h->d_work = nullptr;
  h->work_cap = 0;
  cudaError_t e = cudaMalloc(&h->d_work, n * sizeof(uint64_t));
  if (e == cudaSuccess) h->work_cap = n;
  return e;
}

// Work items of a prefill call whose chunks hold up to `tokens` rows, at most: 256
// rows of a head each, or 128 of two.
size_t work_items_for(const CacheGeom& g, long long tokens) {
  return (size_t)g.B * g.Hq * (size_t)((tokens + 255) / 256);
}

// Before a call that moves the lengths: whether it is being captured.
void note_capture(aoh_cache* h, cudaStream_t s) {
  if (h->captured) return;
  cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(s, &st) != cudaSuccess) {
    cudaGetLastError();  // the legacy stream beside a capture: the launch reports it
    return;
  }
  h->captured = st != cudaStreamCaptureStatusNone;
}

// The H2Share anchor workspace (once per handle; cudaMalloc).
cudaError_t reserve_h2(aoh_cache* h) {
  const CacheGeom& g = h->geom;
  if (g.n_r == 0 || h->d_h2) return cudaSuccess;
  // scores [B][n_r][G][max_seq padded to 4], head states, importance overflow
  cudaError_t e = cudaMalloc(&h->d_h2, h2_workspace_floats(g.B, g.n_r, g.G, g.max_seq) * sizeof(float));
  if (e != cudaSuccess) h->d_h2 = nullptr;
  return e;
}

}  // namespace

extern "C" {

int32_t aoh_version(void) { return 102; }

const char* aoh_last_error(void) { return g_last_error.c_str(); }

size_t aoh_cache_bytes(const aoh_config* cfg, const uint8_t* head_labels) {
  int n_r, n_s;
  if (check_config(cfg, head_labels, &n_r, &n_s) != AOH_OK) return 0;
  return bytes_for(*cfg, n_r, n_s);
}

aoh_status aoh_cache_init(const aoh_config* cfg, const uint8_t* head_labels, void* kv_buffer,
                          size_t kv_buffer_bytes, aoh_cache** out) {
  if (!out) return fail(AOH_ERR_INVALID, "out is NULL");
  *out = nullptr;
  int n_r, n_s;
  aoh_status st = check_config(cfg, head_labels, &n_r, &n_s);
  if (st != AOH_OK) return st;
  const aoh_config& c = *cfg;
  const int G = c.n_q_heads / c.n_kv_heads;
  if (!decode_supported(c.d_head, G))
    return fail(AOH_ERR_UNSUPPORTED, "group size %d with d_head %d is not compiled", G, c.d_head);
  if (!kv_buffer) return fail(AOH_ERR_INVALID, "kv_buffer is NULL");
  if (!aligned(kv_buffer, 256)) return fail(AOH_ERR_INVALID, "kv_buffer must be 256-byte aligned");
  const size_t need = bytes_for(c, n_r, n_s);
  if (kv_buffer_bytes < need)
    return fail(AOH_ERR_CAPACITY, "kv_buffer has %zu bytes, the cache needs %zu", kv_buffer_bytes, need);

  aoh_cache* h = new aoh_cache();
  h->cfg = c;
  h->labels.assign(head_labels, head_labels + c.n_kv_heads);
  h->kv = kv_buffer;
  h->kv_bytes = need;
  h->lens.assign(c.batch, 0);
  CacheGeom& g = h->geom;
  g.B = c.batch;
  g.Hq = c.n_q_heads;
  g.Hkv = c.n_kv_heads;
  g.D = c.d_head;
  g.G = G;
  g.max_seq = c.max_seq;
  g.S = c.sink;
  g.W = c.window;
  g.K = c.chunk;
  g.n_r = n_r;
  g.n_s = n_s;
  int ir = 0, is = 0;
  for (int k = 0; k < c.n_kv_heads; ++k) {
    g.kind[k] = head_labels[k];
    if (head_labels[k] == AOH_RETRIEVAL) {
      g.idx[k] = (uint8_t)ir;
      g.r_head[ir++] = (uint8_t)k;
    } else {
      g.idx[k] = (uint8_t)is;
      g.s_head[is++] = (uint8_t)k;
    }
  }

  cudaError_t e = cudaGetDevice(&h->device);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&h->num_sms, cudaDevAttrMultiProcessorCount, h->device);
  if (e != cudaSuccess) {
    delete h;
    return cuda_fail(e, "cudaGetDevice");
  }
  const size_t n_lens = ((size_t)c.batch + 63) / 64 * 64;
  const size_t n_cnt = ((size_t)c.batch * c.n_kv_heads + 63) / 64 * 64;
  const size_t n_part = decode_partial_floats(2 * h->num_sms, G, c.d_head);
  const size_t n_gcnt = ((size_t)4 * h->num_sms + 63) / 64 * 64;
  const size_t meta_bytes = (2 * n_lens + n_cnt + n_gcnt + 64) * 4 + n_part * 4;
  e = cudaMalloc(&h->meta, meta_bytes);
  if (e == cudaSuccess) e = cudaMemset(h->meta, 0, meta_bytes);
  if (e == cudaSuccess) e = cudaDeviceSynchronize();
  if (e != cudaSuccess) {
    if (h->meta) cudaFree(h->meta);
    delete h;
    return cuda_fail(e, "metadata allocation");
  }
  uint32_t* base = static_cast<uint32_t*>(h->meta);
  h->d_lens = reinterpret_cast<int32_t*>(base);
  h->d_chunk = reinterpret_cast<int32_t*>(base + n_lens);
  h->d_counters = base + 2 * n_lens;
  h->d_gcounters = h->d_counters + n_cnt;
  h->d_done = h->d_gcounters + n_gcnt;
  h->d_err = h->d_done + 32;
  h->d_partials = reinterpret_cast<float*>(base + 2 * n_lens + n_cnt + n_gcnt + 64);
  if (!make_decode_maps(&h->maps, h->geom, h->kv)) {
    cudaFree(h->meta);
    delete h;
    return fail(AOH_ERR_CUDA, "cuTensorMapEncodeTiled failed for the cache regions");
  }
  // the prefill work list for the longest chunk a retrieval head can take
  // (max_seq tokens), so that prefill calls within it allocate nothing
  e = reserve_work(h, work_items_for(h->geom, c.max_seq));
  if (e != cudaSuccess) {
    cudaFree(h->meta);
    delete h;
    return cuda_fail(e, "work list allocation");
  }
  *out = h;
  return AOH_OK;
}

aoh_status aoh_cache_reserve(aoh_cache* cache, int32_t max_tokens, int32_t anchor_workspace) {
  if (!cache) return fail(AOH_ERR_INVALID, "cache is NULL");
  if (max_tokens < 0) return fail(AOH_ERR_INVALID, "max_tokens must be >= 0");
  cudaError_t e = reserve_work(cache, work_items_for(cache->geom, max_tokens));
  if (e != cudaSuccess) return cuda_fail(e, "work list allocation");
  if (anchor_workspace) {
    if (!decode_uses_tc(cache->geom.D, cache->geom.G))
      return fail(AOH_ERR_UNSUPPORTED, "the anchor step needs the d_head 128 tensor-core decode");
    e = reserve_h2(cache);
    if (e != cudaSuccess) return cuda_fail(e, "anchor workspace allocation");
  }
  return AOH_OK;
}

void aoh_cache_destroy(aoh_cache* cache) {
  if (!cache) return;
  if (cache->meta) cudaFree(cache->meta);
  if (cache->d_work) cudaFree(cache->d_work);
  if (cache->d_h2) cudaFree(cache->d_h2);
  delete cache;
}

aoh_status aoh_cache_lens(const aoh_cache* cache, int32_t* lens_out) {
  if (!cache || !lens_out) return fail(AOH_ERR_INVALID, "NULL argument");
  std::copy(cache->lens.begin(), cache->lens.end(), lens_out);
  return AOH_OK;
}

aoh_status aoh_cache_region(const aoh_cache* cache, int32_t b, int32_t kv_head, size_t* k_offset,
                            size_t* v_offset, int32_t* capacity) {
  if (!cache || !k_offset || !v_offset || !capacity) return fail(AOH_ERR_INVALID, "NULL argument");
  const CacheGeom& g = cache->geom;
  if (b < 0 || b >= g.B || kv_head < 0 || kv_head >= g.Hkv) return fail(AOH_ERR_INVALID, "b or kv_head out of range");
  const size_t elem = g.region(b, kv_head);
  *capacity = g.capacity(kv_head);
  *k_offset = elem * 2;
  *v_offset = (elem + (size_t)(*capacity) * g.D) * 2;
  return AOH_OK;
}

aoh_status aoh_cache_reset(aoh_cache* cache, void* stream) {
  if (!cache) return fail(AOH_ERR_INVALID, "cache is NULL");
  note_capture(cache, (cudaStream_t)stream);
  std::fill(cache->lens.begin(), cache->lens.end(), 0);
  cudaError_t e = cudaMemsetAsync(cache->d_lens, 0, sizeof(int32_t) * cache->geom.B, (cudaStream_t)stream);
  if (e != cudaSuccess) return cuda_fail(e, "cudaMemsetAsync");
  return AOH_OK;
}

aoh_status aoh_cache_check(aoh_cache* cache, void* stream) {
  if (!cache) return fail(AOH_ERR_INVALID, "cache is NULL");
  cudaError_t e = cudaStreamSynchronize((cudaStream_t)stream);
  if (e != cudaSuccess) return cuda_fail(e, "cudaStreamSynchronize");
  uint32_t err = 0;
  e = cudaMemcpy(&err, cache->d_err, sizeof(err), cudaMemcpyDeviceToHost);
  if (e != cudaSuccess) return cuda_fail(e, "cudaMemcpy");
  if (err) {
    const uint32_t zero = 0;
    cudaMemcpy(cache->d_err, &zero, sizeof(zero), cudaMemcpyHostToDevice);
    if (err & kErrTimeout) return fail(AOH_ERR_TIMEOUT, "a kernel's bounded wait ran out (error word 0x%x)", err);
    return fail(AOH_ERR_CAPACITY,
                "a step or chunk found a sequence whose max_seq tokens leave no room for it (error word 0x%x)", err);
  }
  return AOH_OK;
}

aoh_status aoh_cache_selftest_wait(aoh_cache* cache, int64_t limit_ns, int64_t* elapsed_ns, void* stream) {
  if (!cache) return fail(AOH_ERR_INVALID, "cache is NULL");
  if (limit_ns < 1000000 || limit_ns > 2000000000LL)
    return fail(AOH_ERR_INVALID, "limit_ns must be in [1 ms, 2 s]");
  cudaStream_t s = (cudaStream_t)stream;
  // the elapsed time is staged in the metadata block's spare word after the error word
  unsigned long long* d_elapsed = reinterpret_cast<unsigned long long*>(cache->d_err + 8);
  cudaError_t e = launch_wait_selftest(cache->d_err, (uint64_t)limit_ns, d_elapsed, s);
  if (e != cudaSuccess) return cuda_fail(e, "self-test kernel launch");
  unsigned long long el = 0;
  e = cudaMemcpyAsync(&el, d_elapsed, sizeof(el), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) return cuda_fail(e, "self-test read back");
  if (elapsed_ns) *elapsed_ns = (int64_t)el;
  return AOH_OK;
}

aoh_status aoh_prefill(const void* q, const void* k, const void* v, int32_t T, const int32_t* seq_lens,
                       aoh_cache* cache, void* out, void* stream) {
  if (!cache) return fail(AOH_ERR_INVALID, "cache is NULL");
  if (!k || !v) return fail(AOH_ERR_INVALID, "k and v must not be NULL");
  if (out && !q) return fail(AOH_ERR_INVALID, "q must not be NULL when out is given");
  if (!aligned(k, 16) || !aligned(v, 16) || (q && !aligned(q, 16)) || (out && !aligned(out, 16)))
    return fail(AOH_ERR_INVALID, "q, k, v and out must be 16-byte aligned");
  const CacheGeom& g = cache->geom;
  if (T < 1) return fail(AOH_ERR_INVALID, "T must be >= 1");
  std::vector<int32_t> clen(g.B, T);
  if (seq_lens) {
    for (int b = 0; b < g.B; ++b) {
      if (seq_lens[b] < 1 || seq_lens[b] > T)
        return fail(AOH_ERR_INVALID, "seq_lens[%d] = %d is outside [1, T]", b, seq_lens[b]);
      clen[b] = seq_lens[b];
    }
  }
  const std::vector<int32_t> base = cache->lens;
  if (g.K > 0)
    for (int b = 0; b < g.B; ++b)
      if (base[b] % g.K)
        return fail(AOH_ERR_INVALID, "sequence %d holds %d tokens, not a multiple of chunk %d", b, base[b], g.K);
  std::vector<int32_t> lens(g.B);
  bool chunked = false;
  for (int b = 0; b < g.B; ++b) {
    lens[b] = base[b] + clen[b];
    chunked |= base[b] > 0;
    if (g.n_r > 0 && lens[b] > g.max_seq)
      return fail(AOH_ERR_CAPACITY, "sequence %d would hold %d tokens; max_seq is %d", b, lens[b], g.max_seq);
  }
  cudaStream_t s = (cudaStream_t)stream;
  cudaError_t e = cudaSuccess;
  note_capture(cache, s);
  ChunkLens cl;
  const bool rows_by_value = g.B <= ChunkLens::kMost;
  const bool by_value = rows_by_value && !cache->captured;
  cl.lens = rows_by_value ? nullptr : cache->d_chunk;
  cl.base = by_value ? nullptr : cache->d_lens;
  if (rows_by_value) {
    for (int b = 0; b < g.B; ++b) cl.by_value[b] = make_int2(clen[b], base[b]);
  } else {
    e = cudaMemcpyAsync(cache->d_chunk, clen.data(), sizeof(int32_t) * g.B, cudaMemcpyHostToDevice, s);
    if (e != cudaSuccess) return cuda_fail(e, "cudaMemcpyAsync(chunk lengths)");
  }

  // attention first: a chunk's own writes to a streaming ring would overwrite
  // positions its rows still read
  if (out) {
    const float scale_log2 = (float)(1.4426950408889634 / sqrt((double)g.D));
    std::vector<int> costs;
    const std::vector<uint64_t> items = prefill_schedule(g, base, clen, &costs);
    const std::vector<uint64_t> pairs = prefill_pairs(items, costs, cache->num_sms);
    // up to kPrefillByValue items travel as kernel arguments: a copy from
    // pageable memory waits for the stream's earlier work, so the GPU would
    // stand idle from one call to the next
    if (items.size() > (size_t)kPrefillByValue) {
      e = reserve_work(cache, items.size());
      if (e != cudaSuccess) return cuda_fail(e, "work list allocation");
      e = cudaMemcpyAsync(cache->d_work, items.data(), items.size() * sizeof(uint64_t), cudaMemcpyHostToDevice, s);
      if (e != cudaSuccess) return cuda_fail(e, "cudaMemcpyAsync(work)");
    }
    PrefillTcArgs pa;
    memset(&pa, 0, sizeof(pa));
    pa.geom = g;
    pa.out = out;
    pa.chunk = cl;
    pa.work = cache->d_work;
    pa.err = cache->d_err;
    pa.T = T;
    pa.scale_log2 = scale_log2;
    if (!prefill_tc_make_maps(&pa, q, k, v, g.B, T))
      return fail(AOH_ERR_CUDA, "cuTensorMapEncodeTiled failed for q/k/v");
    if ((chunked || cache->captured) && !prefill_tc_make_cache_maps(&pa, cache->kv))
      return fail(AOH_ERR_CUDA, "cuTensorMapEncodeTiled failed for the cache");
    e = pairs.empty() && prefill_is_short(costs, cache->num_sms) ? launch_prefill_short(pa, items, cache->num_sms, s)
                                                                 : launch_prefill_tc(pa, items, pairs, s);
    if (e != cudaSuccess) return cuda_fail(e, "prefill kernel launch");
  }

  AppendArgs ap;
  ap.geom = g;
  ap.k = k;
  ap.v = v;
  ap.kv = cache->kv;
  ap.chunk = cl;
  ap.new_lens = by_value ? cache->d_lens : nullptr;
  ap.after_prefill = by_value && out != nullptr;
  ap.T = T;
  e = launch_append(ap, s);
  if (e != cudaSuccess) return cuda_fail(e, "append kernel launch");
  if (!by_value) {
    e = launch_lens_add(cache->d_lens, cl, g, cache->d_err, s);
    if (e != cudaSuccess) return cuda_fail(e, "length update launch");
  }
  cache->lens = lens;
  return AOH_OK;
}

}  // extern "C"

namespace {

// Host checks shared by the decode entry points; fills `a` for the step, the
// longest sequence's rows and the step's total rows (every retrieval row; ring rows of streaming heads).
aoh_status prepare_decode(const void* q, const void* k_new, const void* v_new, aoh_cache* cache, void* out,
                          cudaStream_t s, DecodeArgs& a, long long& total, long long& longest) {
  if (!cache) return fail(AOH_ERR_INVALID, "cache is NULL");
  if (!q || !k_new || !v_new || !out) return fail(AOH_ERR_INVALID, "q, k_new, v_new and out must not be NULL");
  if (!aligned(q, 16) || !aligned(k_new, 16) || !aligned(v_new, 16) || !aligned(out, 16))
    return fail(AOH_ERR_INVALID, "q, k_new, v_new and out must be 16-byte aligned");
  const CacheGeom& g = cache->geom;
  total = longest = 0;
  for (int b = 0; b < g.B; ++b) {
    if (g.n_r > 0 && cache->lens[b] + 1 > g.max_seq)
      return fail(AOH_ERR_CAPACITY, "sequence %d holds %d tokens; max_seq is %d", b, cache->lens[b], g.max_seq);
    const long long t1 = cache->lens[b] + 1;
    longest = std::max(longest, t1);
    total += g.n_r * t1 + g.n_s * std::min<long long>(t1, g.S + g.W);
  }
  a.tcr = cache->maps.tcr;
  a.tcs = cache->maps.tcs;
  a.tcr_odd = cache->maps.tcr_odd;
  a.tcs_odd = cache->maps.tcs_odd;
  a.geom = g;
  a.q = q;
  a.k_new = k_new;
  a.v_new = v_new;
  a.out = out;
  a.kv = cache->kv;
  a.lens = cache->d_lens;
  a.partials = cache->d_partials;
  a.counters = cache->d_counters;
  a.gcounters = cache->d_gcounters;
  a.done = cache->d_done;
  a.err = cache->d_err;
  a.scale_log2 = (float)(1.4426950408889634 / sqrt((double)g.D));
  note_capture(cache, s);
  return AOH_OK;
}

}  // namespace

extern "C" {

aoh_status aoh_decode_step(const void* q, const void* k_new, const void* v_new, aoh_cache* cache, void* out,
                           void* stream) {
  DecodeArgs a;
  long long total = 0, longest = 0;
  const aoh_status st = prepare_decode(q, k_new, v_new, cache, out, (cudaStream_t)stream, a, total, longest);
  if (st != AOH_OK) return st;
  const CacheGeom& g = cache->geom;
  decode_tc_split(a, g, longest, total, cache->num_sms);
  cudaError_t e = launch_decode_tc(a, (cudaStream_t)stream);
  if (e != cudaSuccess) return cuda_fail(e, "decode kernel launch");
  for (int b = 0; b < g.B; ++b) cache->lens[b] += 1;
  return AOH_OK;
}

aoh_status aoh_decode_step_anchor(const void* q, const void* k_new, const void* v_new, aoh_cache* cache, void* out,
                                  int32_t top_k, int32_t* indices, void* stream) {
  DecodeArgs a;
  long long total = 0, longest = 0;
  const aoh_status st = prepare_decode(q, k_new, v_new, cache, out, (cudaStream_t)stream, a, total, longest);
  if (st != AOH_OK) return st;
  const CacheGeom& g = cache->geom;
  if (top_k < 1) return fail(AOH_ERR_INVALID, "top_k must be >= 1");
  if (g.n_r > 0 && !indices) return fail(AOH_ERR_INVALID, "indices must not be NULL");
  if (!decode_uses_tc(g.D, g.G))
    return fail(AOH_ERR_UNSUPPORTED, "the anchor step needs the d_head 128 tensor-core decode");
  if (g.n_r > 0 && !cache->d_h2) {
    cudaError_t e = reserve_h2(cache);
    if (e != cudaSuccess) return cuda_fail(e, "anchor workspace allocation");
  }
  if (g.n_r > 0) h2_decode_outputs(cache->d_h2, g.B, g.n_r, g.G, g.max_seq, &a.scores, &a.score_stride, &a.score_stats);
  decode_tc_split(a, g, longest, total, cache->num_sms);
  cudaStream_t s = (cudaStream_t)stream;
  cudaError_t e = launch_decode_tc(a, s);
  if (e != cudaSuccess) return cuda_fail(e, "decode kernel launch");
  for (int b = 0; b < g.B; ++b) cache->lens[b] += 1;
  if (g.n_r > 0) {
    e = launch_h2_topk(cache->d_h2, g.max_seq, cache->d_lens, g.B, g.n_r, g.G, top_k, indices, s);
    if (e != cudaSuccess) return cuda_fail(e, "top-k kernel launch");
  }
  return AOH_OK;
}

aoh_status aoh_decode_step_reuse(const void* q, const void* k_new, const void* v_new, aoh_cache* cache, void* out,
                                 const int32_t* indices, int32_t n_anchor_groups, int32_t top_k,
                                 const int32_t* group_map, void* stream) {
  DecodeArgs a;
  long long total = 0, longest = 0;
  const aoh_status st = prepare_decode(q, k_new, v_new, cache, out, (cudaStream_t)stream, a, total, longest);
  if (st != AOH_OK) return st;
  const CacheGeom& g = cache->geom;
  // d_head 128: the tcgen05 kernel's gather warps copy the borrowed rows, a
  // gathered row weighing gather_w / ring_w contiguous rows in the CTA split
  const bool tc = decode_uses_tc(g.D, g.G);
  if (!tc && !decode_cc_supported(g.D, g.G))
    return fail(AOH_ERR_UNSUPPORTED, "group size not compiled for the reuse step");
  if (top_k < 1) return fail(AOH_ERR_INVALID, "top_k must be >= 1");
  if (g.n_r > 0) {
    if (!indices || !group_map) return fail(AOH_ERR_INVALID, "indices and group_map must not be NULL");
    if (!aligned(indices, 4)) return fail(AOH_ERR_INVALID, "indices must be 4-byte aligned");
    if (n_anchor_groups < 1 || n_anchor_groups > kMaxKvHeads)
      return fail(AOH_ERR_INVALID, "n_anchor_groups must be in [1, %d]", kMaxKvHeads);
    for (int i = 0; i < g.n_r; ++i)
      if (group_map[i] < 0 || group_map[i] >= n_anchor_groups)
        return fail(AOH_ERR_INVALID, "group_map[%d] = %d is outside [0, %d)", i, group_map[i], n_anchor_groups);
    for (int i = 0; i < g.n_r; ++i) a.idx_map[i] = (uint8_t)group_map[i];
  }
  a.idx = g.n_r > 0 ? indices : nullptr;
  a.top_k = top_k;
  a.n_idx_groups = n_anchor_groups;
  if (tc) reuse_tc_weights(g.G, &a.gather_w, &a.ring_w);
  // every retrieval item now holds min(top_k, t + 1) rows
  total = 0;
  for (int b = 0; b < g.B; ++b) {
    const long long t1 = cache->lens[b] + 1;
    total += (g.n_r * std::min<long long>(t1, top_k) * a.gather_w +
              g.n_s * std::min<long long>(t1, g.S + g.W) * a.ring_w + a.ring_w - 1) / a.ring_w;
  }
  a.n_ctas = tc ? decode_tc_ctas(total, cache->num_sms) : decode_cc_ctas(total, cache->num_sms);
  cudaError_t e = tc ? launch_decode_tc(a, (cudaStream_t)stream) : launch_decode_cc(a, (cudaStream_t)stream);
  if (e != cudaSuccess) return cuda_fail(e, "reuse decode kernel launch");
  for (int b = 0; b < g.B; ++b) cache->lens[b] += 1;
  return AOH_OK;
}

}  // extern "C"
