"""The host's plan of a prefill call, compiled alone (no GPU): in a launch on
clusters of two CTAs the halves of a shared item meet in one cluster, whatever the
number of SMs, and every item is there once, or as its two halves."""

import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2608_06849_gb300", "csrc")

PROBE = r"""
#include "aoh_api.cu"
int main() {
  int launches = 0, late = 0;
  for (int sms : {5, 9, 12, 13, 76, 151, 152})
    for (int n = 1; n <= 4 * sms + 2; ++n)
      for (int heavy : {1, n / 2, sms, sms + 1, sms + 2, 2 * sms + 1, n - 1})
        for (int light : {3, 47}) {
          if (heavy < 1 || heavy > n) continue;
          std::vector<uint64_t> items;
          std::vector<int> costs;
          for (int i = 0; i < n; ++i) {
            items.push_back(prefill_item(i, i % 64, i));
            costs.push_back(i < heavy ? 94 : light);
          }
          const std::vector<uint64_t> pairs = prefill_pairs(items, costs, sms);
          if (pairs.empty()) continue;
          ++launches;
          if (pairs.size() % 2) return printf("odd list: %d SMs, %d items, %d heavy\n", sms, n, heavy), 1;
          std::vector<int> seen(n, 0);
          bool first_shared = false;
          for (size_t e = 0; e < pairs.size(); e += 2) {
            const bool a = pairs[e] != kPrefillNone && pairs[e] >= kPrefillHalf;
            const bool b = pairs[e + 1] != kPrefillNone && pairs[e + 1] >= kPrefillHalf;
            if (a != b || (a && pairs[e] != pairs[e + 1]))
              return printf("halves apart: %d SMs, %d items, %d heavy\n", sms, n, heavy), 1;
            if (e == 0) first_shared = a;
            late += a && !first_shared;
            for (int k = 0; k < 2; ++k)
              if (pairs[e + k] != kPrefillNone) seen[(pairs[e + k] & ~kPrefillHalf) >> 34] += a ? 1 : 2;
          }
          for (int x : seen)
            if (x != 2) return printf("an item lost or repeated: %d SMs, %d items, %d heavy\n", sms, n, heavy), 1;
        }
  printf("%d launches, %d clusters shared past whole ones\n", launches, late);
  return launches == 0 || late == 0;
}
"""


def test_halves_of_an_item_meet_in_one_cluster(tmp_path):
    src, exe = tmp_path / "probe.cpp", tmp_path / "probe"
    src.write_text(PROBE)
    # the launchers that the plan does not reach are left out of the program
    subprocess.run(["g++", "-std=c++17", "-O1", "-w", "-ffunction-sections", "-I", CSRC, "-I",
                    "/usr/local/cuda/include", str(src), "-o", str(exe), "-Wl,--gc-sections"], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
