"""The FP64 Gram and Q-form at every kind of width: one and several tiles, slot
groups full and ragged, column groups that a ragged n leaves short, row ranges
and panels with remainders, leading dimensions above m.

Elementwise bounds: a k-term FP64 dot product in any order is within (k + 2) eps
of the sum of the magnitudes, and both sides round."""
import numpy as np
import pytest

import oracle
import synth
from gpu_util import EPS, to_dev, to_host

pytestmark = pytest.mark.gpu

WIDTHS = [1, 2, 7, 15, 16, 17, 22, 23, 31, 32, 33, 47, 48, 49, 63, 64, 65, 79, 80, 81, 90, 91, 96, 97, 100, 110, 111,
          112, 113, 126, 127, 128, 129, 130, 143, 160, 161, 200, 255, 256, 257, 300, 385, 400, 513]


@pytest.fixture(scope="module")
def cq():
    import paper_1710_08471_gb300 as cq

    return cq


def _with_ld(A, pad):
    import torch

    m, n = A.shape
    buf = torch.full((n, m + pad), float("nan"), dtype=torch.float64, device="cuda")
    x = buf[:, :m].t()
    x.copy_(to_dev(A))
    return x


@pytest.mark.parametrize("n", WIDTHS)
def test_syrk_and_qform(cq, n):
    g = np.random.default_rng(n)
    for m, pad in ((n, 0), (n + 37, 5), (2000 + n, 1)):
        A = g.standard_normal((m, n))
        dA = _with_ld(A, pad)
        with cq.Plan(m, n) as p:
            W = to_host(p.syrk(dA))
            assert np.array_equal(W, W.T)
            assert np.all(np.abs(W - A.T @ A) <= 2 * (m + 2) * EPS * (np.abs(A).T @ np.abs(A)))
            Ri = np.triu(g.standard_normal((n, n)))
            Q = to_host(p.qform(dA, to_dev(Ri)))
            assert np.all(np.abs(Q - A @ Ri) <= 2 * (n + 2) * EPS * (np.abs(A) @ np.abs(Ri)))


@pytest.mark.parametrize("n", [n for n in WIDTHS if n <= 128])
def test_fused_matches_plain(cq, n):
    """Both orders of summation, held to the FP64 tolerances."""
    for m in (n, 3 * n + 50, 20011):
        kappa = 1e3 if m > 2 * n else None
        A = synth.make_matrix(m, n, kappa, seed=n) if m > n else np.eye(n) + 0.5 * np.triu(np.ones((n, n))) / n
        for fused in (False, True):
            with cq.Plan(m, n, fused=fused) as p:
                Q, R, info = p.factor(to_dev(A))
            assert info.status == 0
            Q, R = to_host(Q), to_host(R)
            assert oracle.orthogonality(Q) <= 1e-12 and oracle.residual(A, Q, R) <= 1e-13
            assert np.array_equal(np.tril(R, -1), np.zeros((n, n)))
