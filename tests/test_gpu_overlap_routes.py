"""Overlap of small bases (one launch) and of large ones (two launches): the same shells alone and as one of many far-apart
copies, every class to (8, 8), contracted and not, coincident centres, against each other and the oracle at the parity bar."""
import os

import numpy as np
import pytest

import oracle
from paper_2404_16245_gb300 import workloads as W
from tests import parity

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

THREADS = os.cpu_count() or 1


@pytest.mark.parametrize("ls,nprim,copies", [(list(range(9)), 1, 30), (list(range(9)), 3, 16), ([0], 1, 900), ([2, 2], 8, 40),
                                             ([8, 0, 8], 2, 24)])
def test_alone_and_among_copies(ls, nprim, copies):
    from paper_2404_16245_gb300 import shgo
    rng = np.random.default_rng(len(ls) + nprim)
    sites = rng.uniform(0.0, 2.0, (2, 3))
    exps = np.exp(rng.uniform(np.log(0.3), np.log(6.0), len(ls) * nprim))
    coefs = rng.uniform(0.2, 1.0, len(ls) * nprim)
    xyz = np.array([sites[i % 2] for i in range(len(ls))])
    one = W.make_basis(ls, [nprim] * len(ls), exps, coefs, xyz)
    shift = 60.0 * np.stack(np.unravel_index(np.arange(copies), (10, 10, 10)), 1)
    many = W.make_basis(ls * copies, [nprim] * (len(ls) * copies), np.tile(exps, copies), np.tile(coefs, copies),
                        (shift[:, None] + xyz[None]).reshape(-1, 3))

    def S(basis):
        H = shgo.Basis(basis)
        out = shgo.overlap(H).cpu().numpy()
        H.close()
        assert np.array_equal(out, out.T)
        return out

    ref, small, large = oracle.overlap(one, threads=THREADS, precision="ld"), S(one), S(many)
    parity.check(small, ref, what="alone")
    n = ref.shape[0]
    parity.check(large[:n, :n], ref, what="first of the copies")
    assert not large[:n, n:].any()
