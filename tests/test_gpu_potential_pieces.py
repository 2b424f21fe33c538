"""The potential's weights in many pieces (SHGO_ESP_SCRATCH_DOUBLES) against one piece per class.

Points add their pieces' sums in any order: within 1e-13 of the largest value, some hundred roundings of 2^-53."""
import numpy as np
import pytest

from paper_2404_16245_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("cap", [1, 3000, 100000])
def test_pieces(monkeypatch, cap):
    from paper_2404_16245_gb300 import shgo
    rng = np.random.default_rng(cap)
    basis = W.random_basis(3, 24, 6, max_prim=3, box=3.0, exp_lo=0.1, exp_hi=30.0)
    n = W.nbf(basis)
    D = rng.standard_normal((n, n))
    D = torch.tensor(D + D.T, device="cuda")
    X = torch.tensor(rng.uniform(-4.0, 7.0, (150, 3)), device="cuda")
    H = shgo.Basis(basis)
    want = [shgo.esp(H, D, X), shgo.esp_gradient(H, D, X)]
    monkeypatch.setenv("SHGO_ESP_SCRATCH_DOUBLES", str(cap))
    for f, ref in zip((shgo.esp, shgo.esp_gradient), want):
        got = f(H, D, X)
        assert float((got - ref).abs().max()) <= 1e-13 * float(ref.abs().max())
    H.close()
