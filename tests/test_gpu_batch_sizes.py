"""A batch that needs both sizes of the grouped kernel (n <= 32 and n <= 64) and
planned problems at once, with and without right-hand sides, eager and replayed
from a graph: every problem against the oracle, and bit for bit the same as in
a batch of its own."""
import numpy as np
import pytest

import oracle
import synth
from gpu_util import to_dev, to_host

pytestmark = pytest.mark.gpu

SHAPES = [(40, 1), (300, 8), (1000, 16), (65, 31), (2000, 32), (33, 32), (2000, 33), (500, 48), (64, 64), (3000, 64),
          (3000, 70), (2500, 130)]


@pytest.fixture(scope="module")
def cq():
    import paper_1710_08471_gb300 as cq

    return cq


def _problems(cq, shapes, rhs):
    import torch

    out = []
    for i, (m, n) in enumerate(shapes):
        A = synth.make_matrix(m, n, 1e2 if m > 2 * n else None, seed=i)
        if m <= 2 * n:
            A = A + 8.0 * np.eye(m, n)
        p = [to_dev(A), cq.empty_colmajor(m, n, device="cuda"), cq.empty_colmajor(n, n, device="cuda")]
        if rhs:
            p += [to_dev(synth.make_rhs(m, seed=i)), torch.empty(n, dtype=torch.float64, device="cuda")]
        out.append(tuple(p))
    return out


@pytest.mark.parametrize("rhs", [False, True])
@pytest.mark.parametrize("graph", [False, True])
def test_all_sizes_together(cq, rhs, graph):
    import torch

    probs = _problems(cq, SHAPES, rhs)
    s = torch.cuda.Stream() if graph else None
    torch.cuda.synchronize()
    with cq.Batch(len(probs), small_work_limit=1 << 40, stream=s, graph=graph) as b:
        for _ in range(3 if graph else 1):
            infos = b.factor(probs)
    assert all(i.status == 0 for i in infos)
    for p in probs:
        A, Q, R = (to_host(t) for t in p[:3])
        assert oracle.orthogonality(Q) <= 1e-12 and oracle.residual(A, Q, R) <= 1e-13
        if rhs:
            ref = np.linalg.lstsq(A, to_host(p[3]), rcond=None)[0]
            assert np.linalg.norm(to_host(p[4]) - ref) <= 1e-9 * np.linalg.norm(ref)
        alone = _problems(cq, [A.shape], rhs)[0]
        q = (p[0],) + alone[1:3] + ((p[3], alone[4]) if rhs else ())
        with cq.Batch(1, small_work_limit=1 << 40) as b:
            b.factor([q])
        assert torch.equal(q[1], p[1]) and torch.equal(q[2], p[2])
        if rhs:
            assert torch.equal(q[4], p[4])
