"""The z chunk length of an operator launch (the header's own function, compiled for
the host): the choice over every number of chunks one by one, at a cost that does
not grow with the number of planes."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SRC = r"""
#include <algorithm>
#include <chrono>
#include <cstdio>
#include "rsn_internal.h"
using namespace rsn;
static int one_by_one(int nz, int R, bool fp64, long long columns, int per_sm) {
  int best = 1;
  double best_cost = 1e300;
  for (int zt = 1; zt <= std::max(1, nz / 2); ++zt) {
    const int lz = std::min(kMaxLz, ((nz + zt - 1) / zt + kMuPlanes - 1) / kMuPlanes * kMuPlanes);
    const long long n = columns * ((nz + lz - 1) / lz), wave = 152LL * per_sm;
    const double cost = (double)((n + wave - 1) / wave) * (fp64 ? lz + 0.35 * R + 1.0 : lz + R + 1.5);
    if (cost < best_cost * 0.999) best_cost = cost, best = lz;
  }
  return best;
}
int main() {
  for (int nz = 1; nz <= 700; ++nz)
    for (int R : {1, 4, 6})
      for (int per_sm : {1, 2, 4})
        for (long long columns : {1, 3, 8, 16, 47, 144, 256, 1000, 9000})
          for (bool fp64 : {false, true}) {
            const int got = pick_lz(nz, R, fp64, columns, per_sm), want = one_by_one(nz, R, fp64, columns, per_sm);
            if (got != want) return printf("%d planes, R %d, %lld columns: %d, not %d\n", nz, R, columns, got, want), 1;
          }
  // the longest grids: 2^31 - 1 planes of one point, 2,000 launches
  const auto t0 = std::chrono::steady_clock::now();
  long long sum = 0;
  for (int k = 0; k < 2000; ++k) sum += pick_lz(2147483647 - k, 1 + k % 6, k & 1, 1 + k, 2);
  const double ms = std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - t0).count();
  if (sum < 2000 * kMuPlanes || ms > 1000) return printf("%.1f ms\n", ms), 1;
  return 0;
}
"""


def test_chunk_length(tmp_path):
    cuda = os.path.join(os.path.dirname(os.path.dirname(shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc")), "include")
    if not shutil.which("g++") or not os.path.exists(os.path.join(cuda, "cuda_runtime.h")):
        pytest.skip("needs g++ and the CUDA headers")
    src, exe = tmp_path / "chunks.cpp", tmp_path / "chunks"
    src.write_text(SRC)
    p = subprocess.run(["g++", "-std=c++17", "-O2", "-I", cuda, "-I", os.path.join(ROOT, "paper_1401_0782_gb300", "csrc"),
                        str(src), "-o", str(exe)], capture_output=True, text=True)
    assert p.returncode == 0, p.stderr
    p = subprocess.run([str(exe)], capture_output=True, text=True)
    assert p.returncode == 0, p.stdout + p.stderr
