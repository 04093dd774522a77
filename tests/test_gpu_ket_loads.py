"""FP32 kernels' ket loads (csrc/eri_core.cuh, KetLoads): the next primitive pair
loaded ahead, E non-zeros in 16-byte loads whose last group is partly padding.
Mixed J and K of all s/p/d class pairs against the oracle for one, two and four
primitives a shell, with ket counts that leave tiles partly empty; tolerance as
in the other parity tests, 2e-6 of max|J|."""
import numpy as np
import pytest

from .helpers import random_mol

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_24968_gb300.build import build
    build()


@pytest.mark.parametrize("nprim", [1, 2, 4])
@pytest.mark.parametrize("natom", [1, 3])
@pytest.mark.parametrize("tau", [0.0, 1e-10])
def test_mixed_builds_match_oracle(natom, nprim, tau):
    from oracle import OracleBasis
    from paper_2510_24968_gb300 import FSIM_MIXED, Basis
    rng = np.random.default_rng(100 * natom + nprim)
    mol = random_mol(rng, natom=natom, lmax=2, nprim=nprim)
    gb, ob = Basis(mol), OracleBasis(mol)
    D = rng.standard_normal((gb.nbf, gb.nbf))
    D = D + D.T
    Jo, Ko = ob.jk(D, tau=tau)[:2]
    J, K = gb.fock_build(D, tau=tau, precision=FSIM_MIXED)
    J2 = gb.j_build(D, tau=tau, precision=FSIM_MIXED)
    tol = 2e-6 * np.abs(Jo).max()
    assert np.abs(J - Jo).max() < tol and np.abs(K - Ko).max() < tol and np.abs(J2 - Jo).max() < tol
