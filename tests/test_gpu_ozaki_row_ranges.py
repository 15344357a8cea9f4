"""Split-precision Gram where its row ranges fill the SMs more than four times
(704, 1500 and 1600 columns), from few rows to more than the ranges need, one plan
for several row counts. The bound is the error-free split's own."""
import numpy as np
import pytest

import oracle
import synth
from gpu_util import EPS, to_dev, to_host
from test_gpu_ozaki import frac_bits, pow2_above

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [704, 1500, 1600])
def test_gram_ranges(n):
    import paper_1710_08471_gb300 as cq

    for m in (n, 2 * n + 65, 6001):
        A = synth.make_matrix(m, n, None, seed=m + n)
        absA, ce = np.abs(A), pow2_above(np.max(np.abs(A), axis=0))
        with cq.Plan(m, n, precision=cq.CQR2_OZAKI_BF16) as p:
            W = to_host(p.syrk(to_dev(A)))
        bound = m * np.outer(ce, ce) * 2.0 ** (2 - frac_bits(7)) + 2 * m * EPS * (absA.T @ absA)
        assert np.array_equal(W, W.T) and np.all(np.abs(W - oracle.syrk(A)) <= bound)
    with cq.Plan(6001, n, precision=cq.CQR2_OZAKI_BF16) as p:
        for m in (6001, n, 3 * n + 1):
            A = synth.make_matrix(m, n, 10.0, seed=m)
            Q, R, info = p.factor_rows(to_dev(A))
            assert info.status == 0
            assert oracle.orthogonality(to_host(Q)) <= 1e-11 and oracle.residual(A, to_host(Q), to_host(R)) <= 1e-12
