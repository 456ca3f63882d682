"""One batch context serving maps of 4-slot buckets only, wider ones only and
both in turn (its two sets of kernels, on the same ring slots), over more rounds
than the ring has slots: masks and values equal those of plain calls."""
import pytest
import torch

from paper_2110_00511_gb300 import ash

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("order", [(4,), (16,), (4, 8), (4, 16, 4, 4, 8)])
def test_batches_of_mixed_bucket_sizes(order):
    from paper_2110_00511_gb300 import build
    build.build()
    g = torch.Generator(device="cuda").manual_seed(len(order))

    def keys(n, dim):
        return torch.randint(-40, 40, (n, dim), generator=g, device="cuda", dtype=torch.int32)

    def pair(dim, buckets):
        t = ash.default_tuning()
        t.slots_per_bucket, t.slots_per_capacity = buckets, 1.2
        return [ash.HashMap(dim, 40_000, [(1,)], [torch.float32], tuning=t) for _ in range(2)]

    maps = [(dim, s, *pair(dim, s)) for s in sorted(set(order)) for dim in (1, 2, 3, 4)]
    batch = ash.Batch()
    for r in range(10):
        s = order[r % len(order)]
        use = [m for m in maps if m[1] == s or (s == 8 and r % 2)]
        items, plain = [], []
        for dim, _, batched, single in use:
            ins, fnd, era = keys(3_001, dim), keys(5_000, dim), keys(1_023, dim)
            val = torch.rand((3_001, 1), generator=g, device="cuda")
            items += [(batched, ash.ASH_OP_INSERT, ins, val), (batched, ash.ASH_OP_FIND, fnd, None),
                      (batched, ash.ASH_OP_ERASE, era, None)]
            mask = single.insert(ins, [val])[1]
            idx, found = single.find(fnd)
            plain += [(mask, None), (found, single.gather_values(idx)), (single.erase(era), None)]
        out = batch.run(items)
        for (idx, mask), (want, values), (hm, op, _, _) in zip(out, plain, items):
            assert torch.equal(mask, want)
            if op == ash.ASH_OP_FIND:
                assert torch.equal(hm.gather_values(idx), values)
    for _, _, batched, single in maps:
        a, b = batched.stats(), single.stats()
        assert a["live"] == b["live"] and a["live"] <= a["used_slots"]
