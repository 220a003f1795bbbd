"""aoh_h2share_map when a CUDA call fails after its first launch (the next call may
use the workspace, so the call has to end with the stream synchronised and the
error word cleared), and on several devices of a process. The host code is compiled with a fake of the CUDA runtime that
logs the calls and fails one of them; nothing runs on a GPU."""

import os
import subprocess

import pytest

from paper_2608_06849_gb300 import build as aoh_build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROBE = r"""
#include <stdio.h>
#include <stdlib.h>
#include "h2map.cu"

extern "C" const char* fake_calls();
extern "C" void* fake_memory();
extern "C" const char* fake_attributes();
extern "C" int fail_encode, fail_launch, fake_device;
int fail_encode = -1, fail_launch = -1;

static CUresult encode(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                       const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                       CUtensorMapL2promotion, CUtensorMapFloatOOBfill) {
  static int n = 0;
  return n++ == fail_encode ? CUDA_ERROR_INVALID_VALUE : CUDA_SUCCESS;
}
namespace aoh {
PFN_cuTensorMapEncodeTiled_v12000 encode_fn() { return encode; }
void record_error(const char*) {}
}
int main(int, char** v) {
  fail_encode = atoi(v[1]);
  fail_launch = atoi(v[2]);
  const uint8_t lab[2] = {0, 1};
  int32_t map[2];
  void* w = fake_memory();
  int st = 0;
  for (const char* d = v[3]; *d; ++d) {
    fake_device = *d - '0';
    st = aoh_h2share_map(w, w, w, w, 8, 2, 64, 512, lab, lab, map, nullptr, nullptr);
  }
  printf("%d %s %s\n", st, fake_calls(), fake_attributes());
}
"""

FAKE = r"""
#include <cuda_runtime_api.h>
#include <string.h>
#include <string>

static std::string calls;  // L launch, Z clearing of the error word, C copy back, S synchronise
static char memory[1 << 22];
static int launches = 0;
extern "C" {
extern int fail_launch;
const char* fake_calls() { return calls.c_str(); }
void* fake_memory() { return memory; }
int fake_device = 0;
static std::string attributes;  // the device of each cudaFuncSetAttribute
const char* fake_attributes() { return attributes.c_str(); }
cudaError_t cudaGetDevice(int* d) { return *d = fake_device, cudaSuccess; }
cudaError_t cudaMalloc(void** p, size_t n) { return *p = memory, n <= sizeof(memory) ? cudaSuccess : cudaErrorMemoryAllocation; }
cudaError_t cudaFree(void*) { return cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) {
  attributes += (char)('0' + fake_device);
  return cudaSuccess;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t*, const void*, void**) {
  if (launches++ == fail_launch) return cudaErrorInvalidValue;
  return calls += 'L', cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* p, int, size_t n, cudaStream_t) {
  if (p == memory && n == 4) calls += 'Z';
  return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) {
  memcpy(d, s, n);
  return calls += 'C', cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t) { return calls += 'S', cudaSuccess; }
// what the compiler's start-up code and launch stubs name
void** __cudaRegisterFatBinary(void*) { static void* h; return &h; }
char __cudaInitModule(void**) { return 0; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char*, char*, const char*, int, void*, void*, void*, void*, int*) {}
int __cudaGetKernel(void**, const void*) { return 0; }
int __cudaLaunchKernel(void*, dim3, dim3, void**, size_t, cudaStream_t) { return 0; }
int __cudaPopCallConfiguration(dim3*, dim3*, size_t*, void*) { return 0; }
cudaError_t cudaLaunchKernel(const void*, dim3, dim3, void**, size_t, cudaStream_t) { return cudaSuccess; }
}
"""


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    d = tmp_path_factory.mktemp("h2map")
    (d / "probe.cu").write_text(PROBE)
    (d / "fake.cpp").write_text(FAKE)
    subprocess.run([aoh_build.NVCC, *aoh_build.ARCH, "-std=c++17", "--expt-relaxed-constexpr", "-w", "-cudart", "none", "-I",
                    aoh_build.CSRC, str(d / "probe.cu"), str(d / "fake.cpp"), "-o", str(d / "probe")], check=True)
    return str(d / "probe")


@pytest.mark.parametrize("encode,launch,want", [
    (-1, -1, "0 LLLCS"),   # no failure
    (0, -1, "3 ZS"),       # the key side's maps
    (7, -1, "3 LZS"),      # the query side's, the key side running
    (-1, 1, "3 LZS"),      # the query side's launch
    (-1, 2, "3 LLZS"),     # the mapping's launch
])
def test_a_failed_call_leaves_nothing_running(probe, encode, launch, want):
    r = subprocess.run([probe, str(encode), str(launch), "0"], capture_output=True, text=True, check=True)
    assert " ".join(r.stdout.split()[:2]) == want


def test_attributes_are_set_on_every_device(probe):
    """Kernel attributes belong to a device: set on each device's first launch."""
    r = subprocess.run([probe, "-1", "-1", "01102"], capture_output=True, text=True, check=True)
    st, _, devices = r.stdout.split()
    assert st == "0" and devices == "012"
