"""The primitive-quartet bounds' byte arithmetic (csrc/eri_core.cuh), compiled as a
host program: prim_mask keeps exactly the primitive pairs whose byte is at least
prim_least's, for every count of primitive pairs and every threshold, and a
dropped quartet's bound 2^(ea + eb) never exceeds the threshold 2^lt.
"""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
NVCC = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")

PROGRAM = r"""
#include <cstdio>
#include <cstring>
#include "eri_core.cuh"
using namespace fsim;
int main() {
  long bad = 0, kept = 0;
  unsigned r = 1;
  for (int trial = 0; trial < 400; ++trial) {
    unsigned char by[16];
    for (int k = 0; k < 16; ++k) {
      r = r * 1664525u + 1013904223u;
      by[k] = 0x80 | (trial == 0 ? 127 : (trial == 1 ? 0 : (r >> 24) & 127));
    }
    uint4 v;
    std::memcpy(&v, by, 16);
    for (int npp = 1; npp <= 16; ++npp)
      for (int least = 0; least <= 127; ++least) {
        unsigned want = 0;
        for (int k = 0; k < npp; ++k) want |= (unsigned)((by[k] & 127) >= least) << k;
        bad += prim_mask(v, least, npp) != want;
        kept += want != 0;
      }
  }
  // bytes: 2^(v - 96) bounds the side; dropped only if the product is at most 2^lt
  for (int lt = -200; lt <= 60; ++lt)
    for (int va = 0; va <= 127; ++va)
      for (int vb = 0; vb <= 127; ++vb) {
        const bool drop = vb < prim_least(lt, va);
        if (drop && (va == kPrimNoBound || (va - kPrimBias) + (vb - kPrimBias) > lt)) ++bad;
        if (!drop && va != kPrimNoBound && vb < 127 && (va - kPrimBias) + (vb - kPrimBias) < lt) ++bad;
      }
  for (int va = 0; va <= 127; ++va) bad += prim_least(kPrimKeepAll, va) != 0;
  printf("%ld %ld\n", bad, kept);
  return 0;
}
"""


def test_prim_mask_and_threshold(tmp_path):
    nvcc = NVCC if os.path.exists(NVCC) else shutil.which("nvcc")
    if not nvcc:
        pytest.skip("nvcc not available")
    src, exe = tmp_path / "prim.cu", tmp_path / "prim"
    src.write_text(PROGRAM)
    inc = os.path.join(ROOT, "paper_2510_24968_gb300", "csrc")
    r = subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17", "--expt-relaxed-constexpr",
                        "-I", inc, str(src), "-o", str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    bad, kept = map(int, subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout.split())
    assert bad == 0 and kept > 0
