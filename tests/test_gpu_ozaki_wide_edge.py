"""Split precision on stress inputs at the widths of the 64-column Q-form tile (and
beside them at a width of the 32-column one): spiked, graded, tiny and huge columns
end to end, six slices routed to seven among them, and NaN and infinities in a
column step by step, all with leading dimensions above m (the rows between stay as
they were). Bounds as in test_gpu_ozaki_edge.py."""
import numpy as np
import pytest

import oracle
import synth
from gpu_util import EPS, to_dev, to_host
from test_gpu_ozaki_edge import _kappa_equilibrated, frac_bits, pow2_above

pytestmark = pytest.mark.gpu

PAD = 7


@pytest.fixture(scope="module")
def cq():
    import paper_1710_08471_gb300 as m

    return m


def _padded(cq, rows, cols, A=None):
    """A rows x cols view with leading dimension rows + PAD, and its whole."""
    whole = cq.empty_colmajor(rows + PAD, cols, device="cuda")
    whole.fill_(-3.0)
    if A is not None:
        whole[:rows].copy_(to_dev(A))
    return whole[:rows], whole


def _input(kind, m, n):
    if kind == "graded":
        return synth.graded_rows(m, n, 1e3, seed=n)
    if kind == "spiked":
        return synth.spiked_column(m, n, 1e2, seed=n, col=n - 3)
    A = synth.scaled_column(m, n, 1e2, seed=n, col=n // 2, scale=1e-20)
    return A * np.where(np.arange(n) == 3, 1e15, 1.0)[None, :]


@pytest.mark.parametrize("prec", [1, 2])
@pytest.mark.parametrize("kind", ["graded", "spiked", "scaled"])
@pytest.mark.parametrize("m,n", [(3001, 200), (3001, 250), (3000, 384), (4001, 512)])
def test_stress_inputs(cq, m, n, kind, prec):
    A = np.asfortranarray(_input(kind, m, n))
    k = _kappa_equilibrated(A)
    dA, _ = _padded(cq, m, n, A)
    Q, Qw = _padded(cq, m, n)
    R, Rw = _padded(cq, n, n)
    with cq.Plan(m, n, precision=prec) as p:
        info = p.factor(dA, Q, R)[2]
        used = p.split_slices()
    assert info.status == 0 and (used == 7 or (prec == 2 and kind == "scaled"))
    assert bool((Qw[m:] == -3.0).all()) and bool((Rw[n:] == -3.0).all())
    Q, R = to_host(Q), to_host(R)
    Qo, Ro = oracle.cqr2(A)
    assert oracle.orthogonality(Q) <= max(1e-11, 10 * oracle.orthogonality(Qo))
    assert oracle.residual(A, Q, R) <= max(1e-12, 10 * oracle.residual(A, Qo, Ro))
    assert np.max(np.linalg.norm(R - Ro, axis=0) / np.linalg.norm(Ro, axis=0)) <= 1e-11 * k


@pytest.mark.parametrize("S,prec", [(7, 1), (6, 2)])
@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
@pytest.mark.parametrize("m,n", [(1001, 200), (1001, 250), (700, 384), (1500, 512)])
def test_non_finite_columns(cq, m, n, bad, S, prec):
    g = np.random.default_rng(n)
    A = synth.make_matrix(m, n, None, seed=n)
    A[m // 2, n // 3] = bad
    Ri = np.triu(g.standard_normal((n, n)))
    Ri[n // 3, n - 2] = 0.0  # a later column that the bad one does not enter
    dA, _ = _padded(cq, m, n, A)
    dRi, _ = _padded(cq, n, n, Ri)
    Q, Qw = _padded(cq, m, n)
    W, Ww = _padded(cq, n, n)
    with cq.Plan(m, n, precision=prec) as p:
        p.syrk(dA, W)
        p.qform(dA, dRi, Q)
        Qf, Rf = cq.empty_colmajor(m, n, device="cuda"), cq.empty_colmajor(n, n, device="cuda")
        with pytest.raises(cq.N.CQR2Error):
            p.factor(dA, Qf, Rf)
    assert bool((Qw[m:] == -3.0).all()) and bool((Ww[n:] == -3.0).all())
    W, Q = to_host(W), to_host(Q)
    j = np.arange(n)
    fine = (j < n // 3) | (j == n - 2)
    assert np.all(np.isnan(W[n // 3])) and np.all(np.isnan(W[:, n // 3]))
    ok = np.ix_(j != n // 3, j != n // 3)
    B = np.where(np.isfinite(A), A, 0.0)
    absB, ce = np.abs(B), pow2_above(np.max(np.abs(B), axis=0))
    wb = m * np.outer(ce, ce) * 2.0 ** (2 - frac_bits(S)) + 2 * m * EPS * (absB.T @ absB)
    assert np.all(np.abs(W - B.T @ B)[ok] <= wb[ok])
    assert np.all(np.isnan(Q[:, ~fine]))
    C = B.copy()
    C[:, n // 3] = 0.0  # enters none of the columns looked at
    fe = pow2_above(np.max(ce[:, None] * np.abs(Ri), axis=0))
    qb = n * fe[None, :] * 2.0 ** (2 - frac_bits(S)) + 2 * n * EPS * (np.abs(C) @ np.abs(Ri))
    assert np.all(np.abs(Q - C @ Ri)[:, fine] <= qb[:, fine])
