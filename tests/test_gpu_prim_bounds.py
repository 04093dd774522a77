"""The bounds behind the primitive quartets that are left out (prim_bound_kernel of
csrc/basis.cu, prim_theta of csrc/eri_core.cuh): each primitive pair's byte against the
CPU oracle's Schwarz bound of the same primitives as shells of their own, for s to f
shells from one centre to 13 bohr apart; and that builds at the usual thresholds do
leave primitive quartets out.  The bytes are read from the handle by a small program
compiled against the library's own header.
"""
import math
import os
import subprocess

import numpy as np
import pytest

from .helpers import make_mol

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PKG = os.path.join(ROOT, "paper_2510_24968_gb300")
NVCC = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")

PROGRAM = r"""
#include <cstdio>
#include "fsim_internal.h"
using namespace fsim;
int main() {  // stdin: natom, x y z each; nshell, atom l nprim and alpha coef pairs each
  int na, ns;
  if (scanf("%d", &na) != 1) return 1;
  std::vector<fsim_atom> at(na);
  for (auto& a : at) {
    a.Z = 1;
    for (double& x : a.xyz) if (scanf("%lf", &x) != 1) return 1;
  }
  if (scanf("%d", &ns) != 1) return 1;
  std::vector<fsim_shell_desc> sh(ns);
  std::vector<std::vector<double>> al(ns), co(ns);
  for (int s = 0; s < ns; ++s) {
    if (scanf("%d %d %d", &sh[s].atom, &sh[s].l, &sh[s].nprim) != 3) return 1;
    al[s].resize(4);
    co[s].resize(4);
    for (int k = 0; k < sh[s].nprim; ++k) if (scanf("%lf %lf", &al[s][k], &co[s][k]) != 2) return 1;
    sh[s].alpha = al[s].data();
    sh[s].coef = co[s].data();
  }
  fsim_basis* b = nullptr;
  if (fsim_basis_create(at.data(), na, sh.data(), ns, &b) != FSIM_OK || fsim_schwarz(b, nullptr) != FSIM_OK) return 1;
  for (auto& C : b->cls) {
    std::vector<unsigned char> ub(16 * (size_t)C.n);
    if (C.n && cudaMemcpy(ub.data(), C.ub, ub.size(), cudaMemcpyDeviceToHost) != cudaSuccess) return 1;
    for (int j = 0; j < C.n; ++j)
      for (int k = 0; k < C.h_npp[j]; ++k)
        printf("%d %d %d %d %.17g\n", C.h_idx[j].z, C.h_idx[j].w, k, (int)ub[16 * (size_t)j + k], C.h_Q[j]);
  }
  fsim_basis_destroy(b);
  return 0;
}
"""


def _chain(nprims, lmax):
    atoms = [(1, (3.2 * a, 0.11 * a * a, -0.07 * a)) for a in range(5)]
    sh = []
    for a in range(5):
        for l in range((1, 0, lmax, 1, 0)[a] + 1):
            n = nprims[(a + l) % len(nprims)]
            sh.append((a, l, tuple(0.25 * (1 + 0.1 * l) * 4.0 ** k for k in range(n)), (0.5, -0.6, 0.3, 0.2)[:n]))
    return make_mol(atoms, sh)


def _bytes(mol, tmp_path):
    src, exe = tmp_path / "ub.cu", tmp_path / "ub"
    if not exe.exists():
        src.write_text(PROGRAM)
        r = subprocess.run([NVCC, "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17", "--expt-relaxed-constexpr",
                            "-I", os.path.join(PKG, "csrc"), "-I", os.path.join(ROOT, "include"), str(src), "-o", str(exe),
                            "-L", PKG, "-lfsim", "-Xlinker", "-rpath=" + PKG], capture_output=True, text=True)
        assert r.returncode == 0, r.stderr
    text = [str(mol.natom)] + [" ".join(repr(float(x)) for x in r) for r in mol.xyz] + [str(len(mol.shells))]
    for s in mol.shells:
        text.append(f"{s.atom} {s.l} {len(s.alpha)} " + " ".join(f"{a!r} {c!r}" for a, c in zip(s.alpha, s.coef)))
    r = subprocess.run([str(exe)], input="\n".join(text), capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return [(int(a), int(b), int(k), int(v), float(q)) for a, b, k, v, q in map(str.split, r.stdout.splitlines())]


@pytest.mark.parametrize("nprims", [(1,), (3,), (4, 2, 3, 1)])
@pytest.mark.parametrize("lmax", [2, 3])
def test_bytes_bound_each_primitive_pair(nprims, lmax, tmp_path):
    from oracle import OracleBasis
    from paper_2510_24968_gb300.build import build
    build()
    mol = _chain(nprims, lmax)
    # every primitive a shell of its own; its weight in the contracted shell
    single, first, weight = [], [], []
    for s in mol.shells:
        first.append(len(single))
        S = sum(c * d * (2 * math.sqrt(a * b) / (a + b)) ** (s.l + 1.5) for a, c in zip(s.alpha, s.coef)
                for b, d in zip(s.alpha, s.coef))
        for a, c in zip(s.alpha, s.coef):
            single.append((s.atom, s.l, (a,), (1.0,)))
            weight.append(abs(c) / math.sqrt(S))
    q1 = OracleBasis(make_mol([(1, tuple(x)) for x in mol.xyz], single)).schwarz()
    rows = _bytes(mol, tmp_path)
    assert len(rows) == sum(len(s.alpha) * len(t.alpha) for i, s in enumerate(mol.shells) for t in mol.shells[:i + 1])
    pair = {}
    for a, b, k, byte, Q in rows:
        nb = len(mol.shells[b].alpha)
        x, y = first[a] + k // nb, first[b] + k % nb
        q = q1[x, y] * weight[x] * weight[y]
        assert byte & 0x80
        e = (byte & 0x7f) - 96
        assert q < 2.0 ** e * (1 + 1e-12), (a, b, k)
        if e > -96:
            assert q >= 2.0 ** (e - 1) * (1 - 1e-6), (a, b, k)
        pair.setdefault((a, b), [Q]).append(e)
    # what builds at the usual thresholds leave out of this molecule's kept quartets
    for tau in (1e-9, 1e-11):
        for rel, cap in ((-61, min(tau * 2.0 ** -20, 2.0 ** -53)), (-32, min(tau * 2.0 ** -13, 2.0 ** -43))):
            out = total = 0
            for Q1, *e1 in pair.values():
                for Q2, *e2 in pair.values():
                    if Q1 * Q2 < tau:
                        continue
                    theta = min(math.floor(math.log2(cap)), math.floor(math.log2(Q1)) + math.floor(math.log2(Q2)) + rel)
                    drop = [x + y for x in e1 for y in e2 if x + y <= theta]
                    out, total = out + len(drop), total + len(e1) * len(e2)
                    assert sum(2.0 ** d for d in drop) <= 256 * 2.0 ** rel * Q1 * Q2
            assert out > 0.02 * total or nprims == (1,), (tau, rel, out, total)
