"""A graph plan whose panel width changes captures anew: the graph of the earlier
width uses workspaces that are freed with it."""
import numpy as np
import pytest

import synth
from gpu_util import to_dev, to_host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,n", [(900, 300), (700, 129)])
def test_panel_width_changes_under_a_graph(m, n):
    import torch

    import paper_1710_08471_gb300 as cq

    A = to_dev(synth.make_matrix(m, n, 10.0, seed=n))
    ref = {}
    for b in (0, 64, 128):
        with cq.Plan(m, n) as p:
            p.set_panel_width(b)
            ref[b] = [to_host(t) for t in p.factor(A)[:2]]
    s = torch.cuda.Stream()
    torch.cuda.synchronize()
    with cq.Plan(m, n, stream=s, graph=True) as p:
        Q, R = cq.empty_colmajor(m, n, device="cuda"), cq.empty_colmajor(n, n, device="cuda")
        for b in (128, 0, 64, 128, 0):
            p.set_panel_width(b)
            for _ in range(2):  # capture, replay
                Q.zero_()
                torch.cuda.synchronize()
                p.factor(A, Q, R)
                torch.cuda.synchronize()
                assert np.array_equal(to_host(Q), ref[b][0]) and np.array_equal(to_host(R), ref[b][1])
