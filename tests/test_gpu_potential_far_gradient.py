"""Gradient of the potential at points far from a charge distribution: the field of its lowest multipole.

Shells (l, 0) on one centre have a density of degree l alone, so that far away phi(x) = q(x) / |x|^{2l+1} with q homogeneous
of degree l: x . grad phi = -(l + 1) phi, and for l = 1, q = m . x, grad phi = m / |x|^3 - 3 (m . x) x / |x|^5.

Bar: 1e-13 of the largest gradient.  Every value takes some tens of roundings of 2^-53 (weights, rotation, harmonics, 1/|x|),
and p |x|^2 runs up to 4e4."""
import numpy as np
import pytest

from paper_2404_16245_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("l", [0, 1, 2, 3, 5, 8])
@pytest.mark.parametrize("p,r", [(100.0, 20.0), (2.0, 20.0), (2000.0, 3.0)])
def test_far_gradient(l, p, r):
    from paper_2404_16245_gb300 import shgo
    rng = np.random.default_rng(l)
    basis = W.make_basis([l, 0], [1, 1], [0.6 * p, 0.4 * p], [1.0, 1.0], [np.zeros(3), np.zeros(3)])
    n = 2 * l + 1
    D = np.zeros((n + 1, n + 1))
    D[:n, n] = D[n, :n] = rng.standard_normal(n)
    u = np.concatenate([np.eye(3), rng.standard_normal((61, 3))])
    X = r * u / np.linalg.norm(u, axis=1, keepdims=True)
    H = shgo.Basis(basis)
    Dd, Xd = torch.tensor(D, device="cuda"), torch.tensor(X, device="cuda")
    phi, grad = shgo.esp(H, Dd, Xd).cpu().numpy(), shgo.esp_gradient(H, Dd, Xd).cpu().numpy()
    H.close()
    top = np.linalg.norm(grad, axis=1).max()
    err = np.abs((X * grad).sum(1) + (l + 1) * phi).max() / r
    if l == 1:
        m = phi[:3] * r * r
        ref = m / r ** 3 - 3.0 * (X @ m)[:, None] * X / r ** 5
        err = max(err, np.abs(grad - ref).max())
    assert top > 0.0 and err <= 1e-13 * top, f"{err / top:.2e} of the largest gradient"
