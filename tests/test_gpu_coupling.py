"""The coupling kernel's kinds of nuclei (near, far, on the pair axis) and chunk edges, against the oracle.

Bar per element: 1e-11 |y| + 1e-13 max(1, max |y|) (the parity bar, its absolute part at the scale of the matrix: sums
round relative to their largest terms).  Two one-primitive shells, so that T = p |C - P|^2 is set by the test."""
import os

import numpy as np
import pytest

import oracle
from paper_2404_16245_gb300 import workloads as W
from tests import parity

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

THREADS = os.cpu_count() or 1
# T at which nuclei count as far, per la + lb (rounded values of the kernel's thresholds): both sides are tested
EDGE = {0: 36.5, 1: 40.9, 3: 47.4, 6: 55.4, 11: 66.9, 16: 77.2}


def nuclei(kind, n, p, P, B, lam, rng):
    u = rng.standard_normal((n, 3))
    u /= np.linalg.norm(u, axis=1, keepdims=True)
    if kind == "near":
        return P + rng.uniform(0.0, 3.0, n)[:, None] * u
    if kind == "far":
        return P + rng.uniform(15.0, 60.0, n)[:, None] * u
    if kind == "axis":  # on the line through both centres, some on the centres themselves and far out
        s = np.concatenate([[0.0, 1.0, 2.0, -40.0], rng.uniform(-3.0, 3.0, max(n - 4, 0))])[:n]
        return s[:, None] * B
    if kind == "almost_axis":  # off the line by 1e-3 .. 1e-12
        off = np.outer(10.0 ** rng.uniform(-12, -3, n), np.cross(B, [0.3, 0.5, 0.7]))
        return rng.uniform(-2.0, 3.0, n)[:, None] * B + off
    if kind == "edge":  # T on both sides of the threshold
        T = EDGE[lam] * (1.0 + np.resize([-1e-3, -1e-9, 1e-9, 1e-3, 0.3], n))
        return P + np.sqrt(T / p)[:, None] * u
    mixed = [nuclei(k, n, p, P, B, lam, rng) for k in ("near", "far", "axis", "edge")]
    return np.array([mixed[i % 4][i] for i in range(n)])


@pytest.mark.parametrize("axis", ["z", "general", "same"])
@pytest.mark.parametrize("kind,n", [("near", 1), ("far", 31), ("axis", 7), ("almost_axis", 9), ("edge", 32), ("mixed", 33),
                                    ("mixed", 65)])
def test_kinds_of_nuclei(kind, n, axis):
    from paper_2404_16245_gb300 import shgo
    rng = np.random.default_rng(n)
    for la, lb in ((0, 0), (1, 0), (2, 1), (3, 3), (6, 5), (8, 8)):
        a, b = 0.7, 0.4
        B = {"z": np.array([0.0, 0.0, 1.3]), "general": np.array([0.7, -0.4, 1.1]), "same": np.zeros(3)}[axis]
        P = b / (a + b) * B
        C = nuclei(kind, n, a + b, P, B if axis != "same" else np.array([0.0, 0.0, 1.0]), la + lb, rng)
        Z = rng.uniform(-3.0, 3.0, n)
        Z[n // 2] = 0.0
        basis = W.make_basis([la, lb], [1, 1], [a, b], [1.0, 1.0], [np.zeros(3), B])
        H = shgo.Basis(basis)
        got = shgo.nuclear_attraction(H, torch.tensor(C, device="cuda"), torch.tensor(Z, device="cuda")).cpu().numpy()
        H.close()
        ref = oracle.nuclear_attraction(basis, C, Z, threads=THREADS, precision="ld")
        parity.check(got, ref, atol=parity.ATOL * max(1.0, np.abs(ref).max()), what=f"{kind} {n} {axis} {(la, lb)}")


def test_a_nucleus_without_a_finite_distance_gives_nan():
    from paper_2404_16245_gb300 import shgo
    basis, C, Z = W.config1()
    H = shgo.Basis(basis)
    for bad in (np.nan, np.inf):
        Cb = C.copy()
        Cb[1, 0] = bad
        V = shgo.nuclear_attraction(H, torch.tensor(Cb, device="cuda"), torch.tensor(Z, device="cuda"))
        assert bool(torch.isnan(V).any())
    H.close()
