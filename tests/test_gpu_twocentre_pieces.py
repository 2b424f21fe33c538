"""Overlap and two-centre Coulomb matrices in many pieces and without the table of harmonics
(SHGO_TWOCENTRE_SCRATCH_DOUBLES) against one piece: the same bits."""
import numpy as np
import pytest

from paper_2404_16245_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("cap", [1, 777, 60000])
def test_pieces(monkeypatch, cap):
    from paper_2404_16245_gb300 import shgo
    # 8 sites, so that pairs share their centres; contracted, so that pieces of (a|b) differ in length
    ls = [l for l in range(9) for _ in range(10)]
    rng = np.random.default_rng(9)
    nprim = [1 + i % 3 for i in range(len(ls))]
    sites = rng.uniform(0.0, 3.0, (8, 3))
    sites[1] = sites[0] + [0.0, 0.0, 1.0]
    basis = W.make_basis(ls, nprim, np.exp(rng.uniform(-1.5, 2.0, sum(nprim))), rng.uniform(0.2, 1.0, sum(nprim)),
                         [sites[i % 8] for i in range(len(ls))])
    H = shgo.Basis(basis)
    want = [shgo.overlap(H), shgo.coulomb_2c(H)]
    monkeypatch.setenv("SHGO_TWOCENTRE_SCRATCH_DOUBLES", str(cap))
    got = [shgo.overlap(H), shgo.coulomb_2c(H)]
    H.close()
    for a, b in zip(got, want):
        assert torch.equal(a, b)
