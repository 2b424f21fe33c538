"""The pair kernel's paths against the oracle: shell pairs of one primitive pair (scaled per degree) and of many (contracted
first; more than a chunk of eight, with primitive pairs below the bound among them), few entries and many, and pairs
whose primitive pairs are all skipped.  Parity bar, its absolute part at the scale of the matrix."""
import os

import numpy as np
import pytest

import oracle
from paper_2404_16245_gb300 import workloads as W
from tests import parity

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

THREADS = os.cpu_count() or 1


def basis_of(la, lb, na, nb, sites, rng):
    """One shell la with na primitives on each site and one shell lb with nb."""
    ls, nps, ex, co, xyz = [], [], [], [], []
    for s in sites:
        for l, n in ((la, na), (lb, nb)):
            ls.append(l)
            nps.append(n)
            ex.extend(np.exp(rng.uniform(np.log(0.15), np.log(60.0), n)))
            co.extend(rng.uniform(0.1, 1.0, n) if n > 1 else [1.0])
            xyz.append(s)
    return W.make_basis(ls, nps, ex, co, xyz)


@pytest.mark.parametrize("la,lb", [(0, 0), (1, 0), (1, 1), (2, 0), (3, 2), (4, 4), (6, 1), (8, 7), (8, 8)])
@pytest.mark.parametrize("na,nb", [(1, 1), (1, 2), (3, 3), (5, 7)])
def test_primitive_counts(la, lb, na, nb):
    from paper_2404_16245_gb300 import shgo
    rng = np.random.default_rng(100 * la + 10 * lb + na)
    # two sites near each other, one 4 bohr off: many of its primitive pairs are below the bound
    sites = [[0.0, 0.0, 0.0], [0.4, -0.7, 0.9], [2.5, 2.0, -2.4]]
    basis = basis_of(la, lb, na, nb, sites[:2] if la + lb > 10 else sites, rng)
    C, Z = rng.uniform(-2.0, 2.0, (5, 3)), rng.uniform(1.0, 8.0, 5)
    H = shgo.Basis(basis)
    V = shgo.nuclear_attraction(H, torch.tensor(C, device="cuda"), torch.tensor(Z, device="cuda")).cpu().numpy()
    H.close()
    ref = oracle.nuclear_attraction(basis, C, Z, threads=THREADS, precision="ld")
    parity.check(V, ref, atol=parity.ATOL * max(1.0, np.abs(ref).max()), what=f"{(la, lb)} {(na, nb)}")
    assert np.array_equal(V, V.T)


def test_far_apart_shells_give_zero_blocks():
    from paper_2404_16245_gb300 import shgo
    basis = W.make_basis([3, 2], [2, 2], [1.0, 30.0, 0.8, 5.0], [0.5, 0.5, 0.5, 0.5], [[0, 0, 0], [60.0, 0, 0]])
    H = shgo.Basis(basis)
    V = shgo.nuclear_attraction(H, torch.tensor([[0.0, 0.0, 1.0]], dtype=torch.float64, device="cuda"),
                                torch.ones(1, dtype=torch.float64, device="cuda")).cpu().numpy()
    H.close()
    assert not V[:7, 7:].any() and V[:7, :7].any()
