"""Launches set up early: back-to-back calls on one stream, their input
overwritten right behind each, give bit for bit what calls with a
synchronization between them give. Sizes on both sides of the grids that are
set up early (half an SM each for the Gram and the Q-form, one for a GEMM) and
through every kernel of the chain."""
import numpy as np
import pytest

import synth
from gpu_util import to_dev

pytestmark = pytest.mark.gpu

CALLS = 12


@pytest.fixture(scope="module")
def cq():
    import paper_1710_08471_gb300 as cq

    return cq


@pytest.mark.parametrize("graph", [False, True])
@pytest.mark.parametrize("m,n,kw", [
    (16, 16, {}), (1024, 16, {}), (2400, 33, {}), (4096, 64, {}), (9000, 64, {"fused": True}), (3000, 100, {}),
    (1200, 129, {}), (2000, 256, {}), (1500, 300, {}), (1300, 640, {}), (3000, 200, {"precision": 1}),
])
def test_back_to_back_matches_synchronized(cq, m, n, kw, graph):
    import torch

    As = [to_dev(synth.make_matrix(m, n, None, seed=17 * k + n)) for k in range(CALLS)]
    b = to_dev(synth.make_rhs(m, seed=n))
    with cq.Plan(m, n, graph=graph, **kw) as p:
        A, Q = cq.empty_colmajor(m, n, device="cuda"), cq.empty_colmajor(m, n, device="cuda")
        R, x = cq.empty_colmajor(n, n, device="cuda"), torch.empty(n, dtype=torch.float64, device="cuda")
        ref = []
        for Ak in As:
            A.copy_(Ak)
            torch.cuda.synchronize()
            p.lstsq(A, b, Q, R, x)
            torch.cuda.synchronize()
            ref.append([t.clone() for t in (Q, R, x)])
        torch.cuda.synchronize()
        got = []
        for Ak in As:
            A.copy_(Ak)
            p.lstsq(A, b, Q, R, x, sync=False)
            got.append([t.clone() for t in (Q, R, x)])
        torch.cuda.synchronize()
    for r, g in zip(ref, got):
        for u, v in zip(r, g):
            assert np.array_equal(u.cpu().numpy(), v.cpu().numpy())
