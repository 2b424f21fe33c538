"""The potential kernel's near and far points and block edges (128 points a block, lists of 32), against the oracle.

Bar per point, as in test_gpu_esp: 1e-11 of sum_ab |D_ab V_ab| (gradient: the field integrals') + 1e-13."""
import os

import numpy as np
import pytest

import oracle
from paper_2404_16245_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

THREADS = os.cpu_count() or 1


def points(kind, n, box, rng):
    u = rng.standard_normal((n, 3))
    u /= np.linalg.norm(u, axis=1, keepdims=True)
    r = {"near": rng.uniform(0.0, 2.0, n), "far": rng.uniform(60.0, 200.0, n),
         "mixed": 10.0 ** rng.uniform(-9, 3, n)}[kind]
    return box + r[:, None] * u


@pytest.mark.parametrize("kind,n", [("near", 1), ("near", 33), ("far", 31), ("far", 129), ("mixed", 127), ("mixed", 128),
                                    ("mixed", 161)])
def test_points(kind, n):
    from paper_2404_16245_gb300 import shgo
    rng = np.random.default_rng(n)
    basis = W.make_basis([8, 3, 0, 1], [1, 2, 1, 3], [0.6, 0.3, 2.0, 0.15, 0.2, 1.1, 40.0], [1.0, 0.4, 0.7, 1.0, 0.3, 0.5, 0.2],
                         [[0, 0, 0], [0.5, 1.0, -0.3], [0, 0, 0], [0.0, 0.0, 2.0]])
    X = points(kind, n, np.array([0.1, 0.2, 0.3]), rng)
    X[0] = 0.0  # on a shell centre
    nbf = W.nbf(basis)
    D = rng.standard_normal((nbf, nbf))
    D = (D + D.T) / 2
    H = shgo.Basis(basis)
    Dd, Xd = torch.tensor(D, device="cuda"), torch.tensor(X, device="cuda")
    phi = shgo.esp(H, Dd, Xd).cpu().numpy()
    grad = shgo.esp_gradient(H, Dd, Xd).cpu().numpy()
    H.close()
    assert phi.shape == (n,) and grad.shape == (n, 3)
    one = np.ones(1)
    for i in sorted(set([0, n - 1] + list(range(0, n, max(1, n // 12))))):
        V = oracle.nuclear_attraction(basis, X[i:i + 1], one, threads=THREADS, precision="ld")
        assert abs(phi[i] - (D * V).sum()) <= 1e-13 + 1e-11 * np.abs(D * V).sum(), i
        F = oracle.nuclear_field(basis, X[i:i + 1], one, threads=THREADS, precision="ld")
        for c in range(3):
            assert abs(grad[i, c] - (D * F[c]).sum()) <= 1e-13 + 1e-11 * np.abs(D * F[c]).sum(), (i, c)
