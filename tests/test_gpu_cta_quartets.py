"""J/K through the CTA-per-quartet kernel (csrc/generic.cu) and the FP64 Boys
function at the sizes where they can go wrong: one to four primitives per shell
(1 to 16 primitive pairs, groups and shares of every remainder, the largest
(ff|ff) layout), few and many quartets (shares of a quartet's bra primitive
pairs), and centres far enough apart that T lies on both sides of the table's
end.  Against the oracle with the tolerances of the other parity tests: 1e-10
for the FP64-accurate builds, 2e-6 of max|J| for mixed ones.
"""
import numpy as np
import pytest

from .helpers import make_mol

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _mol(nprims, lmax, natom, spread, seed):
    rng = np.random.default_rng(seed)
    atoms = [(6, tuple(rng.uniform(-spread, spread, 3))) for _ in range(natom)]
    sh = []
    for a in range(natom):
        for l in range(lmax + 1):
            n = nprims[(a + l) % len(nprims)]
            sh.append((a, l, tuple(sorted(rng.uniform(0.25, 2.5, n))), tuple(rng.uniform(0.3, 1.0, n))))
    return make_mol(atoms, sh)


@pytest.mark.parametrize("nprims,lmax,natom,spread", [((1,), 3, 2, 1.5), ((4,), 3, 2, 1.5), ((1, 4, 2, 3), 3, 2, 2.0),
                                                      ((3,), 2, 3, 6.0), ((2, 3), 1, 7, 8.0), ((4, 1), 2, 4, 3.0)])
def test_jk_against_oracle(nprims, lmax, natom, spread):
    from oracle import OracleBasis
    from paper_2510_24968_gb300 import FSIM_DFLOAT, FSIM_FP64, FSIM_MIXED, Basis
    mol = _mol(nprims, lmax, natom, spread, 11 * natom + lmax)
    gb, ob = Basis(mol), OracleBasis(mol)
    D = np.random.default_rng(5).standard_normal((gb.nbf, gb.nbf))
    D = D + D.T
    Jo, Ko, nq = ob.jk(D, tau=1e-11)
    for prec in (FSIM_FP64, FSIM_DFLOAT, FSIM_MIXED):
        J, K = gb.fock_build(D, tau=1e-11, precision=prec)
        assert gb.last_quartet_count() == nq
        tol = 1e-10 if prec != FSIM_MIXED else 2e-6 * np.abs(Jo).max()
        assert np.abs(J - Jo).max() < tol and np.abs(K - Ko).max() < tol, prec
