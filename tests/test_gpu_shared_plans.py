"""Plans whose calls run beside others' (cqr2_plan_set_shared): the same
factorization up to rounding, through every kernel with a shape of its own there,
at ragged sizes, on both sides of the 32-row ranges; and the switch drops what was
prepared or captured for the other setting."""
import numpy as np
import pytest

import oracle
import synth
from gpu_util import EPS, to_dev, to_host

pytestmark = pytest.mark.gpu

CASES = [(16, 16, {}), (33, 1, {}), (63, 31, {}), (1024, 16, {}), (4097, 64, {}), (9001, 64, {"fused": True}), (3001, 100, {}),
         (1200, 129, {}), (20011, 256, {}), (1500, 300, {}), (1300, 640, {}), (700, 256, {"shifted": True}),
         (5000, 200, {"precision": 1}), (2000, 500, {"precision": 2}), (900, 300, {"panel": 128})]


@pytest.fixture(scope="module")
def cq():
    import paper_1710_08471_gb300 as cq

    return cq


def _plan(cq, m, n, kw, **more):
    kw = dict(kw)
    panel = kw.pop("panel", 0)
    p = cq.Plan(m, n, **kw, **more)
    if panel:
        p.set_panel_width(panel)
    return p


@pytest.mark.parametrize("m,n,kw", CASES)
def test_shared_matches_alone(cq, m, n, kw):
    A, b = synth.make_matrix(m, n, 1e2 if n > 1 else None, seed=m + n), synth.make_rhs(m, seed=n)
    dA, db = to_dev(A), to_dev(b)
    out = []
    for shared in (False, True, True):
        with _plan(cq, m, n, kw) as p:
            p.set_shared(shared)
            Q, R, info = p.factor(dA)
            x, _ = p.lstsq(dA, db)[:2]
            out.append([to_host(t) for t in (Q, R, x)])
        assert info.status == 0
    split = kw.get("precision", 0)
    scale = {0: 1.0, 1: 4.0, 2: 256.0}[split]
    for Q, R, _ in out:  # 20 sqrt(m n) roundings, more for the split products' truncation
        assert oracle.orthogonality(Q) <= scale * 20 * np.sqrt(m * n) * EPS + n * EPS
        assert oracle.residual(A, Q, R) <= scale * 20 * np.sqrt(m * n) * EPS + n * EPS
    assert oracle.rel_error(out[1][1], out[0][1]) <= scale * 1e2 * 40 * np.sqrt(m * n) * EPS
    for u, v in zip(out[1], out[2]):
        assert np.array_equal(u, v)


@pytest.mark.parametrize("m,n,kw", [(3001, 100, {}), (2000, 256, {}), (1500, 300, {}), (900, 300, {"panel": 128})])
def test_switching_with_a_captured_graph(cq, m, n, kw):
    import torch

    dA = to_dev(synth.make_matrix(m, n, 10.0, seed=n))
    ref = {}
    for shared in (False, True):
        with _plan(cq, m, n, kw) as p:
            p.set_shared(shared)
            ref[shared] = [to_host(t) for t in p.factor(dA)[:2]]
    s = torch.cuda.Stream()
    torch.cuda.synchronize()
    with _plan(cq, m, n, kw, stream=s, graph=True) as p:
        Q, R = cq.empty_colmajor(m, n, device="cuda"), cq.empty_colmajor(n, n, device="cuda")
        for shared in (False, True, True, False):
            p.set_shared(shared)
            p.factor(dA, Q, R)
            torch.cuda.synchronize()
            assert np.array_equal(to_host(Q), ref[shared][0]) and np.array_equal(to_host(R), ref[shared][1])
