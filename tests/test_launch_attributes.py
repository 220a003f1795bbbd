"""once_per_device, through which every launcher sets its kernel's attributes
(compiled alone against a fake cudaGetDevice): once a device, again after a failure,
and on every call past the devices it keeps a bit for."""

import glob
import os
import re
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2608_06849_gb300", "csrc")

PROBE = r"""
#include <stdio.h>
#include "internal.h"
static int device = 0;
extern "C" cudaError_t cudaGetDevice(int* d) { return *d = device, device < 0 ? cudaErrorNoDevice : cudaSuccess; }
int main() {
  std::atomic<uint64_t> done{0};
  int sets = 0;
  cudaError_t result = cudaSuccess;
  auto call = [&](int d) { device = d; return aoh::once_per_device(done, [&] { return ++sets, result; }); };
  auto expect = [&](int d, int n, cudaError_t e) {
    const cudaError_t got = call(d);
    if (got != e || sets != n) printf("device %d: %d sets, status %d\n", d, sets, (int)got);
  };
  expect(0, 1, cudaSuccess);
  expect(0, 1, cudaSuccess);
  result = cudaErrorInvalidValue;
  expect(1, 2, cudaErrorInvalidValue);
  result = cudaSuccess;
  expect(1, 3, cudaSuccess);
  expect(1, 3, cudaSuccess);
  expect(63, 4, cudaSuccess);
  expect(63, 4, cudaSuccess);
  expect(64, 5, cudaSuccess);
  expect(64, 6, cudaSuccess);
  expect(0, 6, cudaSuccess);
  expect(-1, 6, cudaErrorNoDevice);
}
"""


def test_attributes_once_a_device(tmp_path):
    src, exe = tmp_path / "probe.cpp", tmp_path / "probe"
    src.write_text(PROBE)
    subprocess.run(["g++", "-std=c++17", "-w", "-I", CSRC, "-I", "/usr/local/cuda/include", str(src), "-o", str(exe)],
                   check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, check=True)
    assert r.stdout == ""


def test_no_launcher_keeps_a_flag_of_its_own():
    for f in glob.glob(os.path.join(CSRC, "*.cu*")):
        assert not re.search(r"static bool \w+ = false", open(f).read()), f
