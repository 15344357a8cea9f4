"""The CholInv leaf (one cluster launch, n <= 128) at the edges of its 8-column
blocks and cluster sizes, with pivots outside the reciprocal's range, and its
breakdown reports in every position of a block.

Tolerances as for every CholInv: L within 10 n kappa(L) eps of the oracle, Y
within 10 n kappa(L)^2 eps."""
import numpy as np
import pytest

import oracle
import synth
from gpu_util import EPS, to_dev, to_host

pytestmark = pytest.mark.gpu

SIZES = [1, 2, 7, 8, 9, 15, 16, 17, 24, 31, 32, 33, 40, 56, 63, 64, 65, 72, 96, 120, 127, 128, 129, 200]


@pytest.fixture(scope="module")
def cq():
    import paper_1710_08471_gb300 as cq

    return cq


def _check(L, Y, Lo, Yo):
    n, kappa = len(Lo), np.linalg.cond(Lo)
    assert np.array_equal(np.triu(L, 1), np.zeros((n, n))) and np.array_equal(np.triu(Y, 1), np.zeros((n, n)))
    assert np.linalg.norm(L - Lo) <= 10 * n * kappa * EPS * np.linalg.norm(Lo)
    assert np.linalg.norm(Y - Yo) <= 10 * n * kappa**2 * EPS * np.linalg.norm(Yo)


@pytest.mark.parametrize("n", SIZES)
def test_leaf_matches_oracle(cq, n):
    W = oracle.syrk(synth.make_matrix(3 * n + 10, n, 1e2, seed=n))
    Lo, Yo = oracle.cholinv(W)
    with cq.Plan(n, n) as p:
        dW = to_dev(W)
        L, Y, info = p.cholinv(dW)
        assert info.status == 0
        _check(to_host(L), to_host(Y), Lo, Yo)
        L2, _, _ = p.cholinv(dW, L=dW)  # W may share storage with an output
        assert np.array_equal(to_host(L2), to_host(L))


@pytest.mark.parametrize("n", [5, 40, 100])
def test_leaf_pivots_out_of_range(cq, n):
    """W = D W0 D with powers of two up to 2^+-505: L = D L0, Y = Y0 D^-1."""
    W0 = oracle.syrk(synth.make_matrix(3 * n + 10, n, 1e2, seed=n))
    Lo, Yo = oracle.cholinv(W0)
    d = 2.0 ** np.array([(0, -505, 505, 3)[j % 4] for j in range(n)])
    W = d[:, None] * W0 * d
    with cq.Plan(n, n) as p:
        L, Y, info = p.cholinv(to_dev(W))
    assert info.status == 0
    _check(to_host(L) / d[:, None], to_host(Y) * d, Lo, Yo)


@pytest.mark.parametrize("n,k", [(8, 0), (8, 7), (13, 9), (64, 0), (64, 31), (64, 63), (100, 8), (128, 127), (200, 130)])
@pytest.mark.parametrize("value", [0.0, -1.0, np.nan, np.inf])
def test_leaf_breakdown(cq, n, k, value):
    W = np.eye(n) + 0.01
    W[k, k] = value if value != 0.0 else W[k, k] - 10.0
    with cq.Plan(n, n) as p:
        with pytest.raises(cq.CQR2Error) as e:
            p.cholinv(to_dev(W))
    assert e.value.status == cq.CQR2_ERR_NOT_SPD and e.value.info.failed_pivot == k
