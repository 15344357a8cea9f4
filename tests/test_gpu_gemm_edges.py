"""The FP64 GEMM's tile sizes, k splits and skipped zero groups, through the
steps that run on it: R = R2 R1 (n > 128), the Q-form (n > 256) and CholInv's
recursion. Elementwise bounds: a k-term FP64 dot product in any order is within
(k + 2) eps of the sum of the magnitudes."""
import numpy as np
import pytest

import oracle
import synth
from gpu_util import EPS, to_dev, to_host

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cq():
    import paper_1710_08471_gb300 as cq

    return cq


@pytest.mark.parametrize("n", [129, 144, 160, 191, 193, 257, 320, 449, 700, 1100])
def test_trmm_upper(cq, n):
    g = np.random.default_rng(n)
    R2, R1 = np.triu(g.standard_normal((n, n))), np.triu(g.standard_normal((n, n)))
    with cq.Plan(n, n) as p:
        R = to_host(p.trmm_upper(to_dev(R2), to_dev(R1)))
    assert np.array_equal(np.tril(R, -1), np.zeros((n, n)))
    assert np.all(np.abs(R - R2 @ R1) <= 2 * (n + 2) * EPS * (np.abs(R2) @ np.abs(R1)) + 1e-300)


@pytest.mark.parametrize("m,n", [(257, 257), (300, 258), (511, 271), (1000, 320), (4097, 321), (6001, 777)])
def test_qform(cq, m, n):
    g = np.random.default_rng(n)
    A, Ri = g.standard_normal((m, n)), np.triu(g.standard_normal((n, n)))
    with cq.Plan(m, n) as p:
        Q = to_host(p.qform(to_dev(A), to_dev(Ri)))
    assert np.all(np.abs(Q - A @ Ri) <= 2 * (n + 2) * EPS * (np.abs(A) @ np.abs(Ri)))


@pytest.mark.parametrize("n", [130, 190, 250, 400, 600])
def test_cholinv_recursion(cq, n):
    W = oracle.syrk(synth.make_matrix(3 * n + 10, n, 1e2, seed=n))
    Lo, Yo = oracle.cholinv(W)
    with cq.Plan(n, n) as p:
        L, Y, info = p.cholinv(to_dev(W))
    kappa = np.linalg.cond(Lo)
    assert info.status == 0
    assert np.linalg.norm(to_host(L) - Lo) <= 10 * n * kappa * EPS * np.linalg.norm(Lo)
    assert np.linalg.norm(to_host(Y) - Yo) <= 10 * n * kappa**2 * EPS * np.linalg.norm(Yo)
