"""Shared-memory layouts of the CTA-per-quartet kernel (csrc/generic.cuh), on the host:
for every class pair with up to 16 primitive pairs a side, in FP32 and FP64, no layout
is larger than the limit every launch asks for, the groups fit the CTA, and the limit
fits the device (227 KB a CTA)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
NVCC = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")

PROGRAM = r"""
#include <cstdio>
#include "fsim_internal.h"
#include "generic.cuh"
using namespace fsim;
template <typename Real>
static void walk(long& bad, unsigned& most) {
  for (int X = 0; X < kNumPairClsAll; ++X)
    for (int Y = 0; Y <= X; ++Y)
      for (int pb = 1; pb <= 16; ++pb)
        for (int pk = 1; pk <= 16; ++pk) {
          const GenLayout y = gen_layout<Real>(pair_cls_la(X), pair_cls_lb(X), pair_cls_la(Y), pair_cls_lb(Y), pb, pk);
          bad += y.bytes > kGenMaxSmem || y.nbg < 1 || y.nkg < 1 || y.nbg > 16 || y.nbg * y.nkg > kGenThreads || y.npad < y.nbg * y.nkg;
          most = y.bytes > most ? y.bytes : most;
        }
}
int main() {
  long bad = kGenMaxSmem > 227 * 1024;
  unsigned most = 0;
  walk<float>(bad, most);
  walk<double>(bad, most);
  printf("%ld %u\n", bad, most);
  return 0;
}
"""


def test_no_layout_exceeds_the_limit(tmp_path):
    nvcc = NVCC if os.path.exists(NVCC) else shutil.which("nvcc")
    if not nvcc:
        pytest.skip("nvcc not available")
    src, exe = tmp_path / "lay.cu", tmp_path / "lay"
    src.write_text(PROGRAM)
    r = subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17", "--expt-relaxed-constexpr",
                        "-I", os.path.join(ROOT, "paper_2510_24968_gb300", "csrc"), "-I", os.path.join(ROOT, "include"),
                        str(src), "-o", str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    bad, most = map(int, subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout.split())
    assert bad == 0 and most > 100 * 1024
