"""The grouped kernel's small size does not hold up the planned problems where the
large size runs too: a batch on one side stream with long problems of the small
size, one of the large size and a planned one takes less time than the first and
the last one after the other."""
import numpy as np
import pytest

import synth
from gpu_util import to_dev, to_host

pytestmark = pytest.mark.gpu


def test_planned_problems_run_beside_the_small_size():
    import torch

    import paper_1710_08471_gb300 as cq

    # two long small-size problems occupy two SMs for milliseconds, a planned
    # problem of little work fits beside them
    def problem(m, n, k):
        return (to_dev(synth.make_matrix(m, n, None, seed=k)), cq.empty_colmajor(m, n, device="cuda"),
                cq.empty_colmajor(n, n, device="cuda"))

    narrow = [problem(150000, 16, 1), problem(150000, 16, 2)]
    wide = [problem(100, 40, 3)]
    planned = [problem(65536, 100, 4)]

    def timed(probs):
        with cq.Batch(len(probs), small_work_limit=150000 * 16 * 16, streams=1) as b:
            t = []
            for _ in range(6):
                e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                torch.cuda.synchronize()
                e0.record()
                b.factor(probs, sync=False)
                e1.record()
                torch.cuda.synchronize()
                t.append(e0.elapsed_time(e1))
            assert all(i.status == 0 for i in b.info())
        return sorted(t)[2]

    t_narrow, t_planned = timed(narrow + wide), timed(planned)
    t_all = timed(narrow + wide + planned)
    assert t_all <= max(t_narrow, t_planned) + 0.5 * min(t_narrow, t_planned)
    ref = [to_host(planned[0][1]), to_host(planned[0][2])]
    timed(planned)
    assert np.array_equal(ref[0], to_host(planned[0][1])) and np.array_equal(ref[1], to_host(planned[0][2]))
