"""A batch without any work asks for no snapshot that never lands: the map's
growth checks go on without synchronising, as they do without such a batch."""
import pytest
import torch

from paper_2110_00511_gb300 import ash

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2110_00511_gb300 import build
    build.build()
    ash.lib()


def _host_syncs(empty_batch):
    """Synchronising growth checks of 60 inserts of present keys into a map that
    is past half of its capacity."""
    n = 60_000
    hm = ash.HashMap(3, n, [(1,)], [torch.float32])
    k = torch.arange(n * 6 // 10, device="cuda", dtype=torch.int32)
    keys = torch.stack([k, k * 3, -k], 1).contiguous()
    vals = torch.zeros((len(k), 1), device="cuda")
    hm.insert(keys, [vals])
    torch.cuda.synchronize()
    batch = ash.Batch()
    if empty_batch:
        none = keys[:0]
        for _ in range(3):
            batch.run([(hm, ash.ASH_OP_ACTIVATE, none, None), (hm, ash.ASH_OP_ERASE, none, None)])
            torch.cuda.synchronize()
    before = hm.stats()["host_syncs"]
    for _ in range(60):
        hm.insert(keys[:12_000].contiguous(), [vals[:12_000]])
        torch.cuda.synchronize()  # every snapshot has landed before the next check
    return hm.stats()["host_syncs"] - before


def test_snapshots_go_on_after_an_empty_batch():
    assert _host_syncs(True) == _host_syncs(False)
