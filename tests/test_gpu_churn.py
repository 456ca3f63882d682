"""Windows of keys that come and go over a map, many times, with plain calls
and batched: every pass finds exactly the keys that are in, the used slots
stay near the live entries without a rebuild, and at the end the whole base
is still there (claims reuse tombstones, erases close probe chains)."""
import pytest
import torch

from paper_2110_00511_gb300 import ash

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2110_00511_gb300 import build
    build.build()
    ash.lib()
    torch.cuda.init()


@pytest.mark.parametrize("dim,buckets,slots,claim_mode,batched", [
    (3, 4, 2.0, 0, False), (3, 4, 2.0, 1, False), (2, 4, 1.5, 2, False), (4, 8, 1.6, 0, False), (1, 16, 1.5, 1, False),
    (7, 4, 2.0, 0, False), (3, 4, 2.0, 0, True), (4, 16, 1.5, 0, True), (1, 8, 1.6, 0, True)])
def test_sliding_window(dim, buckets, slots, claim_mode, batched):
    t = ash.default_tuning()
    t.slots_per_bucket, t.slots_per_capacity, t.claim_mode = buckets, slots, claim_mode
    g = torch.Generator(device="cuda").manual_seed(dim * 100 + buckets)
    base_n, n, passes = 30_000, 9_001, 120
    pool = torch.randperm(base_n + 6 * n, generator=g, device="cuda").to(torch.int32)
    keys = torch.stack([pool // (7 ** j) - j for j in range(dim)], 1) if dim > 1 else pool[:, None]
    if dim > 1:
        keys[:, 0] = pool
    keys = keys.contiguous()
    base, windows = keys[:base_n].contiguous(), [w.contiguous() for w in keys[base_n:].split(n)]
    hm = ash.HashMap(dim, base_n + 2 * n, [(1,)], [torch.int32], tuning=t)
    hm.insert(base, [torch.arange(base_n, dtype=torch.int32, device="cuda")])
    batch = ash.Batch() if batched else None
    ones = torch.full((n, 1), 7, dtype=torch.int32, device="cuda")
    for p in range(passes):
        w = windows[p % len(windows)]
        twice = torch.cat([w, w[: n // 3].flip(0)]).contiguous()  # the later occurrences lose
        vals = torch.cat([ones, ones[: n // 3] + 1]).contiguous()
        queries = torch.cat([base[:5_000], w, windows[(p + 1) % len(windows)]]).contiguous()
        if batched:
            (_, new), (idx, found), (_, gone) = batch.run([(hm, ash.ASH_OP_INSERT, twice, vals),
                                                           (hm, ash.ASH_OP_FIND, queries, None),
                                                           (hm, ash.ASH_OP_ERASE, twice, None)])
        else:
            _, new = hm.insert(twice, [vals])
            idx, found = hm.find(queries)
            gone = hm.erase(twice)
        assert new[:n].all() and not new[n:].any()
        assert gone[:n].all() and not gone[n:].any()
        assert found[:5_000 + n].all() and not found[5_000 + n:].any()
        if p == 0:
            first = idx[:5_000].clone()
        assert torch.equal(idx[:5_000], first)
    stats = hm.stats()
    hm.sync_status()
    assert stats["live"] == base_n and stats["used_slots"] >= base_n
    assert stats["used_slots"] <= base_n + base_n // 4 + n
    idx, mask = hm.find(base)
    assert mask.all() and torch.equal(hm.gather_values(idx).view(-1), torch.arange(base_n, dtype=torch.int32, device="cuda"))
    assert hm.size() == base_n and hm.active_indices().numel() == base_n
