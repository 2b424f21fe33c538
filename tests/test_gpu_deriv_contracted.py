"""Derivative and field matrices of contracted shells (primitive pairs contracted before the coupling, four at a time),
against the oracle.  Bar as in test_gpu_deriv: 1e-11 |y| + 1e-13 max |y| per component's matrix."""
import os

import numpy as np
import pytest

import oracle
from paper_2404_16245_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

THREADS = os.cpu_count() or 1


def close(got, ref, what):
    assert np.all(np.isfinite(got)), what
    for x in range(3):
        bar = 1e-11 * np.abs(ref[x]) + 1e-13 * np.abs(ref[x]).max()
        bad = np.abs(got[x] - ref[x]) > bar
        assert not bad.any(), (what, x, int(bad.sum()), float(np.abs(got[x] - ref[x]).max()))


@pytest.mark.parametrize("la,lb", [(0, 0), (1, 0), (1, 1), (2, 1), (3, 3), (4, 2), (6, 5), (7, 7), (8, 8)])
@pytest.mark.parametrize("na,nb", [(1, 2), (2, 2), (3, 5)])
def test_primitive_counts(la, lb, na, nb):
    from paper_2404_16245_gb300 import shgo
    rng = np.random.default_rng(100 * la + 10 * lb + nb)
    ls, nps, ex, co, xyz = [], [], [], [], []
    for s in ([0.0, 0.0, 0.0], [0.5, -0.6, 0.8]):
        for l, n in ((la, na), (lb, nb)):
            ls.append(l)
            nps.append(n)
            ex.extend(np.exp(rng.uniform(np.log(0.2), np.log(40.0), n)))
            co.extend(rng.uniform(0.1, 1.0, n) if n > 1 else [1.0])
            xyz.append(s)
    basis = W.make_basis(ls, nps, ex, co, xyz)
    C, Z = rng.uniform(-2.0, 2.0, (4, 3)), rng.uniform(1.0, 8.0, 4)
    H = shgo.Basis(basis)
    Cd, Zd = torch.tensor(C, device="cuda"), torch.tensor(Z, device="cuda")
    D = shgo.nuclear_attraction_deriv(H, Cd, Zd).cpu().numpy()
    F = shgo.nuclear_field(H, Cd, Zd).cpu().numpy()
    D2 = shgo.nuclear_attraction_deriv(H, Cd, Zd).cpu().numpy()
    H.close()
    assert np.array_equal(D, D2)
    close(D, oracle.nuclear_deriv(basis, C, Z, threads=THREADS, precision="ld"), f"deriv {(la, lb)} {(na, nb)}")
    ref = sum(Z[i] * oracle.nuclear_field(basis, C[i:i + 1], np.ones(1), threads=THREADS, precision="ld") for i in range(4))
    close(F, ref, f"field {(la, lb)} {(na, nb)}")
