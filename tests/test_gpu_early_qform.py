"""A Q-form grid that is set up early leaves no SM with two of its CTAs: a whole
call with few panels takes about as long as its stages timed one by one (event
records between the stages keep any grid from being set up early)."""
import pytest

import synth
from gpu_util import to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,n", [(512, 256), (2432, 256), (2000, 200), (1024, 144)])
def test_whole_call_against_its_stages(m, n):
    import torch

    import paper_1710_08471_gb300 as cq

    A = to_dev(synth.make_matrix(m, n, None, seed=n))
    Q, R = cq.empty_colmajor(m, n, device="cuda"), cq.empty_colmajor(n, n, device="cuda")
    with cq.Plan(m, n) as p:
        whole = []
        for _ in range(12):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            p.factor(A, Q, R, sync=False)
            b.record()
            torch.cuda.synchronize()
            whole.append(a.elapsed_time(b))
        staged = []
        for _ in range(12):
            p.set_profiling(True)
            p.factor(A, Q, R, sync=False)
            staged.append(sum(t for t, _ in p.stage_times().values()))
            p.set_profiling(False)
    assert sorted(whole)[5] <= 1.25 * sorted(staged)[5]
