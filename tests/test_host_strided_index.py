"""The grid-stride index over a list of cells (`StridedIndex` in
csrc/lbm_internal.cuh) at the largest list a box can have: every entry is
visited once and each thread leaves the list, also where its next index is
beyond 2^31. Compiled as host code; no GPU is needed."""
import os
import subprocess

import pytest

from paper_1708_01613_gb300 import build as B

PROGRAM = r"""
#include <cstdio>
#include "lbm_internal.cuh"
int main() {
  for (unsigned n : {0u, 1u, 255u, 256u, 70001u, 0x7fffffffu})
    for (unsigned threads : {256u, 152u * 6 * 256, 1u << 20}) {
      // a thread's visits: all threads for a short list, those around the last entry's for a long one
      const bool all = n < 100000;
      const unsigned last = n ? (n - 1) % threads : 0, from = all ? 0 : (last > 2 ? last - 2 : 0),
                     to = all ? threads : (last + 3 < threads ? last + 3 : threads);
      unsigned long long visits = 0, expected = 0;
      for (unsigned t = from; t < to; ++t) {
        expected += n > t ? (n - t - 1) / threads + 1 : 0;
        unsigned long long seen = 0;
        for (lbm::StridedIndex k{(int)t, (int)threads, (int)n}; k.in(); k.next())
          if ((unsigned)k.at != t + seen * threads || ++seen > n) return printf("n %u threads %u thread %u\n", n, threads, t), 1;
        visits += seen;
      }
      if (visits != expected || (all && visits != n)) return printf("n %u threads %u visits %llu\n", n, threads, visits), 1;
    }
  return 0;
}
"""


def test_every_entry_once_and_out_of_the_list(tmp_path):
    if not os.path.exists(B.nvcc()):
        pytest.skip("nvcc not available")
    src, exe = tmp_path / "strided.cu", tmp_path / "strided"
    src.write_text(PROGRAM)
    r = subprocess.run([B.nvcc(), "-std=c++17", "-O2", "-I", B.INCLUDE, "-I", B.CSRC, str(src), "-o", str(exe)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    out = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert out.returncode == 0, out.stdout
