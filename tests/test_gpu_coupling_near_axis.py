"""Nuclei next to the line through both centres, alone and with others in one chunk, the pair on z: elements that vanish on
the line are small multiples of the offset.

Bar per element: the parity bar, 1e-11 |y| + 1e-13, not scaled by the matrix (the charges are)."""
import os

import numpy as np
import pytest

import oracle
from paper_2404_16245_gb300 import workloads as W
from tests import parity

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

THREADS = os.cpu_count() or 1


def nuclei(kind, rng):
    """Positions and charges: five nuclei off the line by `off`, for the mixed kinds with another close to P."""
    off = {"ulps": 3e-15, "ulps_mixed": 3e-15, "close": 1e-6, "close_mixed": 1e-6, "wide_mixed": 1e-2}[kind]
    z = np.array([2.0, -1.5, 3.0, 0.9, -2.5])
    t = rng.uniform(0.0, 2.0 * np.pi, 5)
    C = np.stack([off * np.cos(t), off * np.sin(t), z], 1)
    if kind.endswith("mixed"):
        C = np.concatenate([C, [[0.05, -0.04, 0.5]], [[0.0, 0.0, 0.0]]])
    Z = np.full(len(C), 40.0 if kind == "ulps" else 0.5)
    return C, Z


@pytest.mark.parametrize("kind", ["ulps", "ulps_mixed", "close", "close_mixed", "wide_mixed"])
@pytest.mark.parametrize("la,lb", [(1, 0), (3, 2), (6, 5), (8, 8)])
def test_next_to_the_axis(la, lb, kind):
    from paper_2404_16245_gb300 import shgo
    C, Z = nuclei(kind, np.random.default_rng(la + lb))
    basis = W.make_basis([la, lb], [1, 1], [0.7, 0.4], [1.0, 1.0], [np.zeros(3), np.array([0.0, 0.0, 1.1])])
    H = shgo.Basis(basis)
    got = shgo.nuclear_attraction(H, torch.tensor(C, device="cuda"), torch.tensor(Z, device="cuda")).cpu().numpy()
    H.close()
    ref = oracle.nuclear_attraction(basis, C, Z, threads=THREADS, precision="ld")
    zero = np.abs(ref) < 1e-9  # the vanishing elements carry the bar's absolute part; the others' rounding scales with Z
    parity.check(np.where(zero, got, 0.0), np.where(zero, ref, 0.0), what=f"small elements {kind} {(la, lb)}")
    parity.check(got, ref, atol=parity.ATOL * max(1.0, np.abs(ref).max()), what=f"{kind} {(la, lb)}")
