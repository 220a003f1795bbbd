// Prefill cache fill (Sec. 5, "Chunked-Prefill Stage"): a chunk of rows at
// positions Lb .. Lb + len - 1 is appended after Lb cached tokens. Retrieval
// KV heads keep every position; streaming KV heads keep the S sinks and the
// last W positions of the new length, position p >= S going to ring row
// S + (p - S) mod W (overwriting the positions that leave the window).
//
// One CTA copies ROWS token rows of one (sequence, KV head) for K and V.
// Each row is D bf16 = D/8 16-byte chunks; consecutive threads take
// consecutive chunks, so loads and stores are coalesced 16-byte accesses.
//
// After a prefill kernel the launch is a programmatic dependent one: its CTAs copy
// on the SMs that the kernel's last wave leaves idle (a prefill CTA's twelve
// allocated warps of 168 registers leave no room beside it). What that kernel may still read is left
// alone until it has ended: the rings of streaming heads that hold tokens
// already (a retrieval head's cached rows stay, and rows past them are masked
// or zeroed by the reader). The first CTA waits for that kernel in any case and
// then sets the lengths, so the launch ends after it. Eight prompts of up to
// 3K rows (54 MB of K and V): the append (16 us), the length update (2.5 us) and
// the copy of the chunk lengths that came before the prefill were 295 - 264 us of
// the call.
#include <limits.h>

#include "common.cuh"
#include "internal.h"

namespace aoh {
namespace {

using bf16 = __nv_bfloat16;
constexpr int kRows = 64;
constexpr int kThreads = 256;

template <int D>
__global__ void __launch_bounds__(kThreads) append_kernel(const __grid_constant__ AppendArgs a) {
  constexpr int CPR = D / 8;  // 16-byte chunks per row
  constexpr int RPI = kThreads / CPR;
  const CacheGeom& g = a.geom;
  const int b = blockIdx.z, h = blockIdx.y;
  if (blockIdx.x == 0 && h == 0 && b == 0 && a.new_lens != nullptr) {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    for (int i = threadIdx.x; i < g.B; i += kThreads) {
      const int2 c = a.chunk.of(i);
      a.new_lens[i] = c.x + c.y;
    }
  }
  const int2 chunk = a.chunk.of(b);
  const int len = chunk.x, Lb = chunk.y;
  const int newlen = Lb + len;
  // a chunk that does not fit (device lengths past the host's) is left out
  if (g.n_r > 0 && newlen > g.max_seq) return;
  const int r0 = blockIdx.x * kRows;          // chunk rows [r0, r1)
  const int r1 = min(r0 + kRows, len);
  if (r0 >= r1) return;
  const bool streaming = g.kind[h] != 0;
  if (streaming && Lb + r1 <= newlen - g.W && Lb + r0 >= g.S) return;  // rows neither sink nor window
  if (streaming && Lb > 0) asm volatile("griddepcontrol.wait;" ::: "memory");
  const int cap = g.capacity(h);
  uint4* Kd = reinterpret_cast<uint4*>(static_cast<bf16*>(a.kv) + g.region(b, h));
  uint4* Vd = Kd + (size_t)cap * CPR;
  const uint4* Ks = static_cast<const uint4*>(a.k);
  const uint4* Vs = static_cast<const uint4*>(a.v);
  const int ch = threadIdx.x % CPR;
  for (int r = r0 + threadIdx.x / CPR; r < r1; r += RPI) {
    const int p = Lb + r;
    int dst = p;
    if (streaming && p >= g.S) {
      if (p < newlen - g.W) continue;
      dst = g.S + (p - g.S) % g.W;
    }
    const size_t src = (((size_t)b * a.T + r) * g.Hkv + h) * CPR + ch;
    Kd[(size_t)dst * CPR + ch] = Ks[src];
    Vd[(size_t)dst * CPR + ch] = Vs[src];
  }
}

// lens[b] += the chunk's rows, stream-ordered.
__global__ void lens_add_kernel(int32_t* lens, const __grid_constant__ ChunkLens chunk, int B, int most, uint32_t* err) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= B) return;
  const int n = lens[b] + chunk.rows(b);
  if (n > most)
    atomicOr(err, kErrCapacity);
  else
    lens[b] = n;
}

}  // namespace

cudaError_t launch_lens_add(int32_t* lens, const ChunkLens& chunk, const CacheGeom& g, uint32_t* err, cudaStream_t s) {
  lens_add_kernel<<<(g.B + 255) / 256, 256, 0, s>>>(lens, chunk, g.B, g.n_r > 0 ? g.max_seq : INT_MAX, err);
  return cudaGetLastError();
}

cudaError_t launch_append(const AppendArgs& a, cudaStream_t s) {
  dim3 grid((a.T + kRows - 1) / kRows, a.geom.Hkv, a.geom.B);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(kThreads);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = a.after_prefill ? 1 : 0;
  if (a.geom.D == 128) return cudaLaunchKernelEx(&cfg, append_kernel<128>, a);
  if (a.geom.D == 64) return cudaLaunchKernelEx(&cfg, append_kernel<64>, a);
  return cudaErrorInvalidValue;
}

}  // namespace aoh
