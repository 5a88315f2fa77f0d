"""The split of a column of planes among blocks (host logic of the two-step pass): the
same as that of a search over every number of blocks, in a fraction of its time, since a
call of olb_step makes it before its launches.  Compiled with the host compiler."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2307_11752_gb300", "csrc")
CUDA_INC = "/usr/local/cuda/include"

DRIVER = r"""
#include <chrono>
#include <cstdio>
#include "olb_internal.h"
static int64_t every(int nz, int64_t tiles, int64_t sms, int& planes) {
  int64_t best = INT64_MAX;
  for (int n = 1; n <= nz; ++n) {
    const int c = (nz + n - 1) / n;
    const int64_t cost = (tiles * ((nz + c - 1) / c) + sms - 1) / sms * (c + 3);
    if (cost < best) { best = cost; planes = c; }
  }
  return best;
}
template <class F>
static double seconds(F f) {
  const auto t = std::chrono::steady_clock::now();
  for (int k = 0; k < 100; ++k) f(k);
  return std::chrono::duration<double>(std::chrono::steady_clock::now() - t).count();
}
int main() {
  int bad = 0;
  for (int nz = 1; nz <= 1200; nz += 1 + nz / 60)
    for (int64_t tiles : {1, 2, 3, 9, 16, 38, 151, 152, 153, 1000, 65536})
      for (int64_t sms : {1, 132, 148, 152}) {
        int a = -1, b = -1;
        if (olb::plane_split(nz, tiles, sms, a) != every(nz, tiles, sms, b) || a != b) ++bad;
      }
  volatile int64_t sink = 0;
  int c = 0;
  const double fast = seconds([&](int k) { sink = sink + olb::plane_split(65535 - k, 8, 152, c); });
  const double slow = seconds([&](int k) { sink = sink + every(65535 - k, 8, 152, c); });
  std::printf("%d differ, %.2f us against %.2f us\n", bad, fast * 1e4, slow * 1e4);
  return bad != 0 || fast * 20 > slow;
}
"""


@pytest.mark.skipif(not os.path.exists(os.path.join(CUDA_INC, "cuda_runtime.h")) or shutil.which("g++") is None,
                    reason="needs the CUDA headers and g++")
def test_plane_split_equals_the_search_over_every_cut(tmp_path):
    src, exe = tmp_path / "drv.cpp", tmp_path / "drv"
    src.write_text(DRIVER)
    r = subprocess.run(["g++", "-O2", "-std=c++17", "-I", CSRC, "-I", CUDA_INC, str(src), "-o", str(exe)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
