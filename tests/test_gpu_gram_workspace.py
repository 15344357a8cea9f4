"""Workspace of the Gram's partial tiles: room for the ranges that a plan can use
(one CTA per SM at 128 columns), and four times that once it is shared."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,resident", [(16, 3), (63, 3), (64, 2), (90, 2), (91, 1), (128, 1), (256, 1), (1000, 1)])
def test_partials_have_room_for_what_is_used(n, resident):
    import torch

    import paper_1710_08471_gb300 as cq

    sms = torch.cuda.get_device_properties(0).multi_processor_count
    ntile = -(-n // 128)
    T = -(-(-(-n // ntile)) // 16) * 16
    tiles, items = ntile * (ntile + 1) // 2, ntile * (ntile - 1) // 2 + -(-ntile // 2)
    part = 8 * tiles * T * T
    with cq.Plan(1 << 16, n) as p:
        own = p.workspace_bytes
        rest = 8 * (11 * n * n + 16 * n * (n // 16 + 2) + (1 << 16) * n * (n > 256) + 3 * 8 * sms * n) + (1 << 16)
        assert own <= max(1, resident * sms // items) * part + rest
        p.set_shared(True)
        p.set_shared(False)
        p.set_shared(True)
        assert p.workspace_bytes <= own + max(1, 4 * sms // items) * part
