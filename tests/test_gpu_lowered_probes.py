"""max_probes lowered on a filled map: a key that sits further along its chain
is not stored a second time, tombstones before it or not; the call reports the
full table instead."""
import pytest
import torch

from paper_2110_00511_gb300 import ash

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("claim_mode", [1, 2, None])  # None: a batch
@pytest.mark.parametrize("dim,buckets", [(3, 4), (2, 8), (4, 16)])
def test_no_key_is_stored_twice(dim, buckets, claim_mode):
    from paper_2110_00511_gb300 import build
    build.build()
    t = ash.default_tuning()
    t.slots_per_bucket, t.slots_per_capacity, t.max_used_fraction, t.auto_grow = buckets, 1.2, 0.98, 0
    t.claim_mode = claim_mode or 0
    n = 20_000
    hm = ash.HashMap(dim, n, tuning=t)
    g = torch.Generator(device="cuda").manual_seed(dim)
    keys = torch.randperm(n, generator=g, device="cuda").to(torch.int32)
    keys = torch.stack([keys * (j + 1) for j in range(dim)], 1).contiguous()
    assert hm.activate(keys)[1].all()
    gone, kept = keys[: n // 8].contiguous(), keys[n // 8:].contiguous()
    assert hm.erase(gone).all()
    before = hm.stats()
    assert before["used_slots"] > before["live"]  # tombstones, in the home buckets of keys that stayed
    t.max_probes = 1
    hm.set_tuning(t)
    batch = ash.Batch()
    for part in kept.split(400):
        if claim_mode is None:
            (_, new), = batch.run([(hm, ash.ASH_OP_ACTIVATE, part.contiguous(), None)])
        else:
            new = hm.activate(part.contiguous())[1]
        assert not new.any()
    t.max_probes = 0
    hm.set_tuning(t)
    assert hm.stats()["live"] == len(kept)
    rows = hm.gather_keys(hm.active_indices())
    assert len(rows) == len(kept) == len(torch.unique(rows, dim=0))
    with pytest.raises(ash.AshError):  # the keys further along were refused
        hm.sync_status()
