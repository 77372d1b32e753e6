"""Blocks of points of the COCG update and of the projector term: they cover a
system's points once, and no position leaves 32 bits, up to the largest grid that
the library takes (2^31 - 1 points).  The header's own functions, compiled for the
host with overflow checks."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SRC = r"""
#include <cstdio>
#include "rsn_internal.h"
using namespace rsn;
int main() {
  const int sizes[] = {1, 127, 128, 129, 511, 512, 513, 69120, (1 << 30) + 1,
                       2147483647 - 640, 2147483647 - 511, 2147483647 - 128, 2147483647 - 127, 2147483647};
  for (int N : sizes) {
    const int nw = kUpdThreads / 32, asked = upd_ctas(N) * nw, nb = blk_count(N);
    if (asked < nb || asked - nb >= nw) return printf("CTAs of %d\n", N), 1;
    if ((long long)(nb - 1) * kBlkPts >= N || (long long)nb * kBlkPts < N) return printf("blocks of %d\n", N), 1;
    for (int k = nb > 8 ? nb - 8 : 0; k < asked; ++k) {
      const int first = blk_first(k, N), len = blk_len(k, N);
      const long long end = (long long)first + len;
      const bool ok = k < nb ? first == (long long)k * kBlkPts && len > 0 && len <= kBlkPts && (k + 1 < nb ? len == kBlkPts : end == N)
                             : first == N && len == 0;
      if (!ok) return printf("block %d of %d: %d + %d\n", k, N, first, len), 1;
    }
  }
  return 0;
}
"""


def test_block_ranges(tmp_path):
    cuda = os.path.join(os.path.dirname(os.path.dirname(shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc")), "include")
    if not shutil.which("g++") or not os.path.exists(os.path.join(cuda, "cuda_runtime.h")):
        pytest.skip("needs g++ and the CUDA headers")
    src, exe = tmp_path / "ranges.cpp", tmp_path / "ranges"
    src.write_text(SRC)
    cmd = ["g++", "-std=c++17", "-O1", "-fsanitize=undefined", "-fno-sanitize-recover=all", "-I", cuda,
           "-I", os.path.join(ROOT, "paper_1401_0782_gb300", "csrc"), str(src), "-o", str(exe)]
    p = subprocess.run(cmd, capture_output=True, text=True)
    assert p.returncode == 0, p.stderr
    p = subprocess.run([str(exe)], capture_output=True, text=True)
    assert p.returncode == 0, p.stdout + p.stderr
