"""Blocks whose elements come from high degrees alone: shells on one centre (or nearly) with l's far apart and nuclei far
away, where the coupling entries of the low degrees are larger by powers of t = sqrt(p) |C - P| and have no part in the block.

Bar: 1e-11 of the block's own largest element (the parity bar's relative part; the absolute part, 1e-13, is far above these
elements)."""
import os

import numpy as np
import pytest

import oracle
from paper_2404_16245_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

THREADS = os.cpu_count() or 1


@pytest.mark.parametrize("la,lb", [(2, 0), (3, 1), (4, 2), (6, 2), (7, 1), (8, 2), (8, 5)])
@pytest.mark.parametrize("a,b,dist,r", [(60.0, 40.0, 0.0, 20.0), (60.0, 40.0, 1e-3, 20.0), (0.5, 0.3, 0.0, 30.0),
                                        (4000.0, 0.1, 1.0, 60.0)])
def test_block_of_high_degrees(la, lb, a, b, dist, r):
    from paper_2404_16245_gb300 import shgo
    u = np.array([0.48, -0.6, 0.64])  # unit vectors
    B = dist * np.array([-0.36, 0.48, 0.8])
    C = r * u[None]
    basis = W.make_basis([la, lb], [1, 1], [a, b], [1.0, 1.0], [np.zeros(3), B])
    H = shgo.Basis(basis)
    got = shgo.nuclear_attraction(H, torch.tensor(C, device="cuda"), torch.ones(1, dtype=torch.float64, device="cuda"))
    H.close()
    ref = oracle.nuclear_attraction(basis, C, np.ones(1), threads=THREADS, precision="ld")
    n = 2 * la + 1
    err, top = np.abs(got.cpu().numpy() - ref)[:n, n:].max(), np.abs(ref[:n, n:]).max()
    assert top > 0.0 and err <= 1e-11 * top, f"{(la, lb)}: {err / top:.2e} of the largest element"
