"""Split-precision Q-form: an output far smaller than its neighbours in the row
keeps all its bits. One column of R^-1 has a single entry, the row's entry of X
there is 2^-31, and their product 2^-32 + 2^-62 is one of the products that the
scheme keeps exactly, whatever the neighbours' sums of up to n products."""
import numpy as np
import pytest

from gpu_util import to_dev, to_host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,n", [(200, 64), (129, 100), (300, 200), (130, 256), (257, 520)])
def test_small_output_beside_large_ones(m, n):
    import paper_1710_08471_gb300 as cq

    with cq.Plan(max(m, n), n, precision=cq.CQR2_OZAKI_BF16) as p:
        for j in sorted({0, 3, n // 3, n // 2 + 1, n - 2}):
            A = np.full((max(m, n), n), 0.5, order="F")
            A[1:, j] = 2.0**-31
            Ri = np.triu(np.full((n, n), 0.5))
            Ri[:, j] = 0.0
            Ri[j, j] = 0.5 + 2.0**-31
            Q = to_host(p.qform(to_dev(A), to_dev(np.asfortranarray(Ri))))
            assert np.all(Q[1:, j] == 2.0**-32 + 2.0**-62), j
