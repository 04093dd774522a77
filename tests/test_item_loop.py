"""The work-item loop of the persistent quartet kernels (csrc/eri_core.cuh, ItemLoop),
on the host: every item below the count and none past it, for counts up to the most a
plan may hold (2^31 - 1 - 128), where the step past the last item leaves the range of a
signed int; and the kernels have no other item loop."""
import glob
import os
import re
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2510_24968_gb300", "csrc")
NVCC = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")

PROGRAM = r"""
#include <cstdio>
#include "eri_core.cuh"
using namespace fsim;
int main() {
  long bad = 0;
  for (int n : {0, 1, 607, 608, 609, 100000, 2147483647 - 128})
    for (unsigned grid : {1u, 152u, 608u, 2432u})
      for (unsigned first = 0; first < grid; first += 151) {
        if ((unsigned)n < first) continue;
        // the last items of the CTA that starts at `first`
        unsigned start = first + (n - first) / grid * grid;
        if (start >= 3 * grid) start -= 3 * grid;
        const long want = start >= (unsigned)n ? 0 : ((long)n - start + grid - 1) / grid;
        long got = 0;
        for (ItemLoop at(start, grid, n); at.more() && got <= want; at.next()) {
          bad += (int)at.i < 0 || (int)at.i >= n;
          ++got;
        }
        bad += got != want;
      }
  printf("%ld\n", bad);
  return 0;
}
"""


def test_item_loop_ends(tmp_path):
    nvcc = NVCC if os.path.exists(NVCC) else shutil.which("nvcc")
    if not nvcc:
        pytest.skip("nvcc not available")
    src, exe = tmp_path / "loop.cu", tmp_path / "loop"
    src.write_text(PROGRAM)
    r = subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17", "--expt-relaxed-constexpr",
                        "-I", CSRC, str(src), "-o", str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    assert subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout.split() == ["0"]


def test_kernels_use_it():
    for path in glob.glob(os.path.join(CSRC, "*.cu*")):
        assert not re.search(r"for \(int \w+ = blockIdx\.x; \w+ < P\.nitems", open(path).read()), path
