"""The least-squares tail (c = Q^T b in partial sums, blocked back substitution)
at the edges of its column groups, row ranges and 32-column blocks."""
import numpy as np
import pytest

import synth
from gpu_util import EPS, to_dev, to_host

pytestmark = pytest.mark.gpu

SHAPES = [(1, 1), (5, 1), (40, 7), (129, 8), (300, 9), (1023, 31), (1024, 32), (1025, 33), (5000, 64), (4097, 65),
          (3000, 255), (3000, 256), (3000, 257), (2600, 513), (70001, 40)]


@pytest.fixture(scope="module")
def cq():
    import paper_1710_08471_gb300 as cq

    return cq


def _tolerance(A, x, b):
    """Least squares through an n-column QR: relative error within
    20 n eps (kappa + kappa^2 |r| / (|A| |x|)) (Householder's own bound)."""
    sv = np.linalg.svd(A, compute_uv=False)
    kappa = sv[0] / sv[-1]
    r = np.linalg.norm(A @ x - b)
    return 20 * A.shape[1] * EPS * (kappa + kappa**2 * r / (sv[0] * np.linalg.norm(x)))


@pytest.mark.parametrize("m,n", SHAPES)
def test_tail_matches_lapack(cq, m, n):
    A, b = synth.make_matrix(m, n, None, seed=m + n), synth.make_rhs(m, seed=m)
    ref = np.linalg.lstsq(A, b, rcond=None)[0]
    with cq.Plan(m, n) as p:
        x, info = p.lstsq(to_dev(A), to_dev(b))
    assert info.status == 0
    assert np.linalg.norm(to_host(x) - ref) <= _tolerance(A, ref, b) * np.linalg.norm(ref)


def test_tail_tiny_diagonal(cq):
    """R's diagonal near 2^-505, below the range whose reciprocals are used:
    the blocks are solved with divisions. Scaling A by a power of two scales x exactly."""
    m, n = 1000, 70
    A, b = synth.make_matrix(m, n, None, seed=3), synth.make_rhs(m, seed=4)
    ref = np.linalg.lstsq(A, b, rcond=None)[0]
    with cq.Plan(m, n) as p:
        x, info = p.lstsq(to_dev(A * 2.0**-510), to_dev(b))
    assert info.status == 0
    assert np.linalg.norm(to_host(x) * 2.0**-510 - ref) <= _tolerance(A, ref, b) * np.linalg.norm(ref)
