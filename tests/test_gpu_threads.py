"""Builds of separate basis handles from two threads at once (calls on one handle must
not overlap, calls on different handles may).  The launches of a class pair need
between 2 and 90 KB of dynamic shared memory depending on the handle's shells and
primitives, and a kernel's limit belongs to the process: one thread's launch must not
depend on the limit another thread has just asked for.  Each result is compared with
the same handle's result alone; they differ by the order of the FP64 atomics only
(2^-44 of the largest element for the FP64 builds; the FP32 integrals of the mixed
ones are the same bits, summed in another order, so the same bound holds)."""
import threading

import numpy as np
import pytest

from .helpers import random_mol

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("prec_name", ["fp64", "mixed", "j fp64", "j mixed"])
def test_builds_of_two_handles_side_by_side(prec_name):
    from paper_2510_24968_gb300 import FSIM_FP64, FSIM_MIXED, Basis
    prec = FSIM_FP64 if "fp64" in prec_name else FSIM_MIXED
    work = []
    for seed, lmax, nprim in ((1, 2, 4), (2, 2 if "mixed" in prec_name or "j" in prec_name else 0, 1)):
        b = Basis(random_mol(np.random.default_rng(seed), natom=2, lmax=lmax, nprim=nprim))
        d = np.random.default_rng(seed + 10).standard_normal((b.nbf, b.nbf))
        D = torch.from_numpy(d + d.T).cuda()
        s = torch.cuda.Stream()

        def build(b=b, D=D, s=s):
            J, K = torch.zeros_like(D), torch.zeros_like(D)
            s.wait_stream(torch.cuda.default_stream())
            if prec_name.startswith("j"):
                b.j_build(D, J, tau=1e-12, precision=prec, stream=s.cuda_stream)
            else:
                b.fock_build(D, J, K, tau=1e-12, precision=prec, stream=s.cuda_stream)
            s.synchronize()
            return J, K
        build()
        work.append((build, build()))
    torch.cuda.synchronize()
    failed, gate = [], threading.Barrier(2)

    def loop(build, ref):
        gate.wait()
        try:
            for _ in range(400):
                for got, want in zip(build(), ref):
                    if float((got - want).abs().max()) > 2.0 ** -44 * float(ref[0].abs().max()) * want.shape[0]:
                        raise AssertionError("another result beside the other thread's builds")
        except Exception as e:  # noqa: BLE001 - reported by the test's own thread
            failed.append(repr(e))
    th = [threading.Thread(target=loop, args=w) for w in work]
    for t in th:
        t.start()
    for t in th:
        t.join()
    assert not failed, failed
