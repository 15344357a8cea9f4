"""Split-precision Gram and Q-form on pairs of CTAs and on single ones: widths on
both sides of every rule (column tiles that pair up and that do not, ragged last
tiles) and row counts with ragged blocks, few and many row ranges. The bounds are
the error-free split's own (see test_gpu_ozaki.py)."""
import numpy as np
import pytest

import oracle
import synth
from gpu_util import EPS, to_dev, to_host
from test_gpu_ozaki import frac_bits, pow2_above

pytestmark = pytest.mark.gpu

WIDTHS = [1, 16, 31, 32, 33, 63, 64, 65, 95, 96, 97, 127, 128, 129, 160, 192, 193, 200, 224, 256, 257, 320, 385, 448, 640]


@pytest.fixture(scope="module")
def cq():
    import paper_1710_08471_gb300 as cq

    return cq


@pytest.mark.parametrize("S,prec", [(7, 1), (6, 2)])
@pytest.mark.parametrize("n", WIDTHS)
def test_syrk_and_qform(cq, n, S, prec):
    g = np.random.default_rng(n)
    for m in (n, n + 65, 129 + 2 * n, 30000 if n <= 256 else 3000):
        A = synth.make_matrix(m, n, None, seed=m + n)
        absA, ce = np.abs(A), pow2_above(np.max(np.abs(A), axis=0))
        Ri = np.triu(g.standard_normal((n, n)) * 10.0 ** g.uniform(-6, 0, (n, n)))
        with cq.Plan(m, n, precision=prec) as p:
            W = to_host(p.syrk(to_dev(A)))
            Q = to_host(p.qform(to_dev(A), to_dev(Ri)))
        bound = m * np.outer(ce, ce) * 2.0 ** (2 - frac_bits(S)) + 2 * m * EPS * (absA.T @ absA)
        assert np.array_equal(W, W.T) and np.all(np.abs(W - oracle.syrk(A)) <= bound)
        fe = pow2_above(np.max(ce[:, None] * np.abs(Ri), axis=0))
        bound = n * fe[None, :] * 2.0 ** (2 - frac_bits(S)) + 2 * n * EPS * (absA @ np.abs(Ri))
        assert np.all(np.abs(Q - A @ Ri) <= bound)


@pytest.mark.parametrize("n", [64, 96, 128, 200, 320])
def test_in_place_pass(cq, n):
    """The second Q-form overwrites Q1 while the pair reads only its slices."""
    m = 5001
    A = synth.make_matrix(m, n, 1e3, seed=n)
    with cq.Plan(m, n, precision=cq.CQR2_OZAKI_BF16, inplace=True) as p:
        Q1, R1, _ = p.factor(to_dev(A))
        dA = to_dev(A)
        Q2, R2, info = p.factor(dA, Q=dA)
    assert info.status == 0 and np.array_equal(to_host(Q1), to_host(Q2)) and np.array_equal(to_host(R1), to_host(R2))
    assert oracle.orthogonality(to_host(Q1)) <= 1e-11 and oracle.residual(A, to_host(Q1), to_host(R1)) <= 1e-12
