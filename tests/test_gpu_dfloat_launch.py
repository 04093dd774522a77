"""Launch choices of double-float builds (fsim_autotune, fsim_set_launch): the FP64
CTA-per-quartet kernel, which the untuned plan gives the heavy and the few-quartet class
pairs, has a code like every other shape, so that a tuning that has it can be saved and
put back after another choice.  Values against the oracle at 1e-10."""
import numpy as np
import pytest

from .helpers import random_mol

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

PAIRS = [(x, y) for x in range(6) for y in range(x + 1)]


def _close(gb, D, ref, prec):
    J, K = gb.fock_build(D, tau=0.0, precision=prec)
    assert np.abs(J - ref[0]).max() < 1e-10 and np.abs(K - ref[1]).max() < 1e-10


def test_choices_come_back():
    from oracle import OracleBasis
    from paper_2510_24968_gb300 import FSIM_DFLOAT, FSIM_FP64, FSIM_MIXED, Basis, FsimError
    mol = random_mol(np.random.default_rng(31), natom=3, lmax=2, nprim=3)
    gb = Basis(mol)
    D = np.random.default_rng(32).standard_normal((gb.nbf, gb.nbf))
    D = D + D.T
    ref = OracleBasis(mol).jk(D)
    _close(gb, D, ref, FSIM_DFLOAT)
    choice = gb.autotune(tau=0.0, precision=FSIM_DFLOAT)
    assert set(choice) == set(PAIRS)  # every class pair has work here, and a code
    _close(gb, D, ref, FSIM_DFLOAT)
    gb.set_launch({xy: 1011 for xy in PAIRS}, tau=0.0, precision=FSIM_DFLOAT)
    _close(gb, D, ref, FSIM_DFLOAT)
    gb.set_launch({xy: c for xy, (c, _) in choice.items()}, tau=0.0, precision=FSIM_DFLOAT)
    _close(gb, D, ref, FSIM_DFLOAT)
    gb.set_launch({xy: 1000 for xy in PAIRS}, tau=0.0, precision=FSIM_DFLOAT)
    _close(gb, D, ref, FSIM_DFLOAT)
    gb.set_launch({(1, 0): 11}, tau=0.0, precision=FSIM_DFLOAT)  # and away from it again
    _close(gb, D, ref, FSIM_DFLOAT)
    for code, prec in ((-1, FSIM_DFLOAT), (1000, FSIM_FP64), (1000, FSIM_MIXED), (-2, FSIM_FP64), (1001, FSIM_DFLOAT),
                       (1010, FSIM_DFLOAT), (2011, FSIM_DFLOAT), (10, FSIM_FP64)):
        with pytest.raises(FsimError):
            gb.set_launch({(1, 1): code}, tau=0.0, precision=prec)
