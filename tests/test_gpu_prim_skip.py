"""Builds that leave out primitive quartets below the rounding of the integrals
(csrc/eri_core.cuh, prim_mask) against builds that evaluate all of them.

A build at screening threshold tau > 0 skips; at tau = 0 nothing is skipped, so
on a molecule whose quartets all survive tau the two differ by the skipped
primitive quartets only.  Each is below theta = min(2^-20 tau, 2^-53) (FP64,
double-float) or min(2^-13 tau, 2^-43) (mixed), at most 81 per quartet, and an
element of J or K takes at most n^2 |D| of them: 81 n^2 max|D| theta bounds the
difference, beside the rounding of the accumulation itself (2^-50 of max|J|).
The oracle's J and K bound both as in the other parity tests.
"""
import numpy as np
import pytest

from .helpers import make_mol

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_24968_gb300.build import build
    build()


@pytest.mark.parametrize("nprim", [1, 3, 4])
@pytest.mark.parametrize("lmax,gap", [(1, 4.0), (2, 3.0), (3, 3.0)])
def test_skipped_primitives_do_not_show(nprim, lmax, gap):
    from oracle import OracleBasis
    from paper_2510_24968_gb300 import FSIM_DFLOAT, FSIM_FP64, FSIM_MIXED, Basis
    rng = np.random.default_rng(10 * lmax + nprim)
    atoms = [(6, (0.0, 0.0, 0.0)), (7, (gap, 0.3, -0.2)), (8, (0.2, gap, 0.4))][:3 if lmax < 3 else 2]
    sh = [(a, l, tuple(0.25 * 2.6 ** k * (1 + 0.1 * l) for k in range(nprim)), tuple(rng.uniform(0.2, 1.0, nprim)))
          for a in range(len(atoms)) for l in range(lmax + 1)]
    mol = make_mol(atoms, sh)
    gb, ob = Basis(mol), OracleBasis(mol)
    D = rng.standard_normal((gb.nbf, gb.nbf))
    D = D + D.T
    tau = 1e-13
    Jo, Ko, nq0 = ob.jk(D, tau=0.0)
    for prec, theta in ((FSIM_FP64, 2.0 ** -20 * tau), (FSIM_DFLOAT, 2.0 ** -20 * tau), (FSIM_MIXED, 2.0 ** -13 * tau)):
        J0, K0 = gb.fock_build(D, tau=0.0, precision=prec)
        J1, K1 = gb.fock_build(D, tau=tau, precision=prec)
        skipped_quartets = (nq0 - gb.last_quartet_count()) * tau * np.abs(D).max()
        bound = 81 * gb.nbf ** 2 * np.abs(D).max() * theta + 2.0 ** -50 * np.abs(Jo).max() * gb.nbf + skipped_quartets
        if prec == FSIM_MIXED:
            bound += 2e-7 * np.abs(Jo).max() * (skipped_quartets > 0)
        assert np.abs(J1 - J0).max() <= bound and np.abs(K1 - K0).max() <= bound, prec
        tol = 1e-10 if prec != FSIM_MIXED else 2e-6 * np.abs(Jo).max()
        assert np.abs(J1 - Jo).max() < tol and np.abs(K1 - Ko).max() < tol, prec
    if lmax < 3:
        J1 = gb.j_build(D, tau=tau, precision=FSIM_FP64)
        assert np.abs(J1 - Jo).max() < 1e-10
