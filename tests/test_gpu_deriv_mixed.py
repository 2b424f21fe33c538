"""Derivative and field matrices of classes that hold shell pairs of one and of many primitive pairs, which take different
variants of the kernel, on both sides of the lines between these.  Bar as in test_gpu_deriv_contracted."""
import numpy as np
import pytest

import oracle
from paper_2404_16245_gb300 import workloads as W
from tests.test_gpu_deriv_contracted import THREADS, close

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("ls", [(0, 1), (4,), (5, 4), (8, 1)])
@pytest.mark.parametrize("nprim", [(1, 1, 2), (1, 2, 3), (1, 4, 5)])
def test_mixed_counts(ls, nprim):
    from paper_2404_16245_gb300 import shgo
    rng = np.random.default_rng(10 * sum(ls) + sum(nprim))
    sites = rng.uniform(0.0, 1.5, (len(nprim), 3))
    shells = [(l, n, sites[i]) for l in ls for i, n in enumerate(nprim)]
    total = sum(n for _, n, _ in shells)
    basis = W.make_basis([l for l, _, _ in shells], [n for _, n, _ in shells], np.exp(rng.uniform(-1.5, 3.0, total)),
                         rng.uniform(0.2, 1.0, total), [x for _, _, x in shells])
    C, Z = rng.uniform(-1.0, 2.0, (3, 3)), rng.uniform(1.0, 8.0, 3)
    H = shgo.Basis(basis)
    Cd, Zd = torch.tensor(C, device="cuda"), torch.tensor(Z, device="cuda")
    D = shgo.nuclear_attraction_deriv(H, Cd, Zd).cpu().numpy()
    F = shgo.nuclear_field(H, Cd, Zd).cpu().numpy()
    H.close()
    close(D, oracle.nuclear_deriv(basis, C, Z, threads=THREADS, precision="ld"), f"deriv {ls} {nprim}")
    ref = sum(Z[i] * oracle.nuclear_field(basis, C[i:i + 1], np.ones(1), threads=THREADS, precision="ld") for i in range(3))
    close(F, ref, f"field {ls} {nprim}")
