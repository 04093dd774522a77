"""Launch shapes of a batched FP64 build: class pairs with few quartets in the
whole batch give each quartet nine threads where every molecule has nine bra
primitive pairs, one thread otherwise; the launches of a build run on several
streams between a fork and a join.  Against the oracle, with the tolerance of
the FP64 parity tests (1e-10)."""
import numpy as np
import pytest

from fsim_synth import water_cluster, workload

from .helpers import random_mol

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_24968_gb300.build import build
    build()


def _set(kind):
    rng = np.random.default_rng(17)
    if kind == "one":
        return [workload("water")]
    mols = [workload("water"), water_cluster(2, geom_seed=7), random_mol(rng, natom=2, lmax=2, nprim=3)]
    if kind == "few primitives":
        mols.append(random_mol(rng, natom=2, lmax=2, nprim=2))
    return mols


@pytest.mark.parametrize("use_graph", [False, True])
@pytest.mark.parametrize("kind", ["one", "nine", "few primitives"])
def test_fp64_batches_match_oracle(kind, use_graph):
    from oracle import OracleBasis
    from paper_2510_24968_gb300 import FSIM_FP64, Basis, Batch
    mols = _set(kind)
    bases = [Basis(m) for m in mols]
    rng = np.random.default_rng(4)
    H = []
    for b in bases:
        d = rng.standard_normal((b.nbf, b.nbf)) * 0.1
        H.append(d + d.T)
    D = [torch.zeros(h.shape, dtype=torch.float64, device="cuda") for h in H]
    J = [torch.zeros_like(d) for d in D]
    K = [torch.zeros_like(d) for d in D]
    bt = Batch(bases, D, J, K, tau=1e-12)
    ref = [OracleBasis(m).jk(h, tau=1e-12)[:2] for m, h in zip(mols, H)]
    for rep in range(2):  # the second build's densities are written while the first may still run
        for d, h in zip(D, H):
            d.copy_(torch.from_numpy(h * (rep + 1)))
        bt.fock(FSIM_FP64, use_graph=use_graph)
        out = [(j.clone(), k.clone()) for j, k in zip(J, K)]
        for (j, k), (jo, ko) in zip(out, ref):
            assert np.abs(j.cpu().numpy() - (rep + 1) * jo).max() < 1e-10
            assert np.abs(k.cpu().numpy() - (rep + 1) * ko).max() < 1e-10
