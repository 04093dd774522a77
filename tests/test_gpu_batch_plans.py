"""A batch keeps one screening plan per precision on each of its molecules, whatever
launch shape its class pairs take; and builds that are queued behind one another with no
wait between them, plain and as graphs, FP64 and mixed in turn on the same accumulators,
each see their own density.  Against the oracle: 1e-10 in FP64, 2e-6 of max|J| mixed."""
import os
import subprocess

import numpy as np
import pytest

from fsim_synth import water_cluster, workload

from .helpers import random_mol

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PKG = os.path.join(ROOT, "paper_2510_24968_gb300")
NVCC = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")

PROGRAM = r"""
#include <cstdio>
#include "fsim_internal.h"
int main() {
  fsim_atom at[2] = {{1, {0, 0, 0}}, {1, {0, 0, 1.4}}};
  double al[3] = {0.3, 0.9, 3.0}, co[3] = {0.4, 0.5, 0.2};
  fsim_shell_desc sh[4] = {{0, 0, 3, al, co}, {0, 1, 3, al, co}, {1, 0, 3, al, co}, {1, 2, 3, al, co}};
  fsim_basis* b = nullptr;
  if (fsim_basis_create(at, 2, sh, 4, &b) != FSIM_OK) return 1;
  double *D, *J, *K;
  const size_t n2 = sizeof(double) * b->nbf * b->nbf;
  if (cudaMalloc(&D, n2) || cudaMalloc(&J, n2) || cudaMalloc(&K, n2) || cudaMemset(D, 0, n2)) return 1;
  fsim_fock_opts o;
  fsim_fock_opts_default(&o);
  o.ptr_mode = FSIM_PTR_DEVICE;
  fsim_batch* bt = nullptr;
  if (fsim_batch_create(&b, 1, &o, &D, &J, &K, &bt) != FSIM_OK) return 1;
  if (fsim_batch_fock(bt, FSIM_FP64, nullptr, 0) != FSIM_OK || cudaDeviceSynchronize() != cudaSuccess) return 1;
  printf("%d\n", (int)b->plans.size());
  fsim_batch_destroy(bt);
  fsim_basis_destroy(b);
  return 0;
}
"""


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_24968_gb300.build import build
    build()


def test_one_plan_per_precision(tmp_path):
    src, exe = tmp_path / "plans.cu", tmp_path / "plans"
    src.write_text(PROGRAM)
    r = subprocess.run([NVCC, "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17", "--expt-relaxed-constexpr",
                        "-I", os.path.join(PKG, "csrc"), "-I", os.path.join(ROOT, "include"), str(src), "-o", str(exe),
                        "-L", PKG, "-lfsim", "-Xlinker", "-rpath=" + PKG], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout.split() == ["2"], r.stdout + r.stderr


@pytest.mark.parametrize("seed", [1, 2])
def test_builds_queued_without_a_wait(seed):
    from oracle import OracleBasis
    from paper_2510_24968_gb300 import FSIM_FP64, FSIM_MIXED, Basis, Batch
    rng = np.random.default_rng(seed)
    mols = [workload("water"), water_cluster(2, geom_seed=7), random_mol(rng, natom=2, lmax=2, nprim=3),
            water_cluster(3, geom_seed=2)]
    bases = [Basis(m) for m in mols]
    H = []
    for b in bases:
        d = rng.standard_normal((b.nbf, b.nbf)) * 0.1
        H.append(d + d.T)
    ref = [OracleBasis(m).jk(h, tau=1e-12)[:2] for m, h in zip(mols, H)]
    scale = [1.0, -2.0, 0.5, 3.0, -1.0, 4.0]
    given = [[torch.from_numpy(h * f).cuda() for h in H] for f in scale]
    D = [torch.zeros(h.shape, dtype=torch.float64, device="cuda") for h in H]
    J = [torch.zeros_like(d) for d in D]
    K = [torch.zeros_like(d) for d in D]
    bt = Batch(bases, D, J, K, tau=1e-12)
    for prec in (FSIM_FP64, FSIM_MIXED):
        bt.fock(prec, use_graph=True)  # graphs made before the queue, which has no host wait
    torch.cuda.synchronize()
    out, precs = [], []
    for step, new in enumerate(given):
        for d, h in zip(D, new):
            d.copy_(h)
        precs.append(FSIM_MIXED if (step + seed) % 2 else FSIM_FP64)
        bt.fock(precs[-1], use_graph=step % 3 != 1)
        out.append([(j.clone(), k.clone()) for j, k in zip(J, K)])
    for f, prec, got in zip(scale, precs, out):
        for (j, k), (jo, ko) in zip(got, ref):
            tol = 1e-10 * abs(f) if prec == FSIM_FP64 else 2e-6 * abs(f) * np.abs(jo).max()
            assert np.abs(j.cpu().numpy() - f * jo).max() < tol
            assert np.abs(k.cpu().numpy() - f * ko).max() < tol
