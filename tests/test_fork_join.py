"""A build's auxiliary streams are joined to the caller's stream whatever happens
between (csrc/fork_join.h): after a launch that failed, after an event call that
failed, and with no auxiliary stream at all.  Compiled for the host against stand-ins
for the three event calls, which write down what the streams were told; and every
build path that forks goes through it.
"""
import glob
import os
import re
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2510_24968_gb300", "csrc")
CUDA = os.path.dirname(os.path.dirname(os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")))

PROGRAM = r"""
#include <cstdio>
#include <cstring>
#include <string>
#include "fork_join.h"
using namespace fsim;
static std::string ops;
static int calls = 0, fail_at = -1;
static cudaError_t op(char what, void* stream, void* event) {
  if (calls++ == fail_at) return cudaErrorUnknown;
  ops += what;
  ops += (char)('0' + (long)stream);
  ops += (char)('a' + (long)event);
  return cudaSuccess;
}
extern "C" cudaError_t CUDARTAPI cudaEventRecord(cudaEvent_t e, cudaStream_t s) { return op('R', s, e); }
extern "C" cudaError_t CUDARTAPI cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned) { return op('W', s, e); }
int main(int argc, char** argv) {
  const int naux = argv[1][0] - '0', good = argv[2][0] - '0';
  if (argc > 3) fail_at = std::stoi(argv[3]);
  cudaStream_t aux[3] = {(cudaStream_t)1, (cudaStream_t)2, (cudaStream_t)3};
  cudaEvent_t join[3] = {(cudaEvent_t)1, (cudaEvent_t)2, (cudaEvent_t)3};
  int rc = 0;
  const cudaError_t e = fork_join((cudaStream_t)0, naux, aux, (cudaEvent_t)0, join, [&](const cudaStream_t* st) {
    for (int k = 0; k <= naux; ++k) {
      if (k == good) { rc = -2; return; }
      ops += 'L';
      ops += (char)('0' + (long)st[k]);
    }
  });
  printf("%s %d %d\n", ops.c_str(), rc, (int)(e != cudaSuccess));
  return 0;
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    cxx = os.environ.get("CXX", "g++")
    if not shutil.which(cxx) or not os.path.exists(os.path.join(CUDA, "include", "cuda_runtime_api.h")):
        pytest.skip("no C++ compiler or CUDA headers")
    d = tmp_path_factory.mktemp("fork")
    (d / "fork.cpp").write_text(PROGRAM)
    r = subprocess.run([cxx, "-std=c++17", "-I", CSRC, "-I", os.path.join(CUDA, "include"), str(d / "fork.cpp"), "-o",
                        str(d / "fork")], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return str(d / "fork")


def _run(program, *args):
    return subprocess.run([program, *map(str, args)], capture_output=True, text=True, check=True).stdout.split()


@pytest.mark.parametrize("naux", [0, 1, 3])
@pytest.mark.parametrize("good", [0, 1, 2, 9])
def test_streams_are_joined_after_a_failed_launch(program, naux, good):
    fork = "R0a" + "".join(f"W{k}a" for k in range(1, naux + 1))
    launched = "".join(f"L{k}" for k in range(min(good, naux + 1)))
    joined = "".join(f"R{k}{'abcd'[k]}W0{'abcd'[k]}" for k in range(1, naux + 1))
    assert _run(program, naux, good) == [fork + launched + joined, "-2" if good <= naux else "0", "0"]


def test_failed_events_are_reported(program):
    assert _run(program, 3, 9, 0) == ["0", "1"]  # no fork: nothing launched
    assert _run(program, 3, 9, 2) == ["R0aW1a", "0", "1"]
    # a failed join of one stream does not leave the others unjoined
    assert _run(program, 3, 9, 4) == ["R0aW1aW2aW3aL0L1L2L3R2cW0cR3dW0d", "0", "1"]


def test_every_build_path_forks_through_it():
    for path in glob.glob(os.path.join(CSRC, "*.cu")):
        text = open(path).read()
        assert not re.search(r"cudaEventRecord\([^)]*(fork_ev|join_ev)", text), path
