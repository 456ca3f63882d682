"""The launch counter counts a batch's own launches: the table's upload, the
phases that have work, and the snapshots where there are any."""
import pytest
import torch

from paper_2110_00511_gb300 import ash

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ops,launches", [
    ((ash.ASH_OP_FIND,), 2), ((ash.ASH_OP_ACTIVATE,), 3), ((ash.ASH_OP_ERASE,), 3),
    ((ash.ASH_OP_ACTIVATE, ash.ASH_OP_FIND), 4), ((ash.ASH_OP_ACTIVATE, ash.ASH_OP_FIND, ash.ASH_OP_ERASE), 6), ((), 0)])
def test_launches_of_a_batch(ops, launches):
    from paper_2110_00511_gb300 import build
    build.build()
    hm = ash.HashMap(2, 10_000)  # far from half full, and too small for snapshots after erases
    keys = torch.arange(600, device="cuda", dtype=torch.int32).view(300, 2)
    batch = ash.Batch()
    before = ash.ash_kernel_launch_count()
    batch.run([(hm, op, keys, None) for op in ops])
    assert ash.ash_kernel_launch_count() - before == launches


def test_a_snapshot_is_one_more():
    from paper_2110_00511_gb300 import build
    build.build()
    hm = ash.HashMap(2, 1000)
    keys = torch.arange(1400, device="cuda", dtype=torch.int32).view(700, 2)
    before = ash.ash_kernel_launch_count()
    ash.Batch().run([(hm, ash.ASH_OP_ACTIVATE, keys, None)])  # past half of the capacity
    assert ash.ash_kernel_launch_count() - before == 4
