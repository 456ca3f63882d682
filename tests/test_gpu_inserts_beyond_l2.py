"""Inserts with values into tables beyond L2, in input order, where the claim's
grid follows rules of its own per bucket size: more keys than one wave of
blocks takes, with duplicates, in every commit width; the first occurrence
wins and brings its value."""
import pytest
import torch

from paper_2110_00511_gb300 import ash

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("buckets", [4, 8, 16])
@pytest.mark.parametrize("dim,commit_keys", [(3, 1), (3, 2), (5, 1), (8, 4)])
def test_first_occurrences_win(buckets, dim, commit_keys):
    from paper_2110_00511_gb300 import build
    build.build()
    t = ash.default_tuning()
    t.slots_per_bucket, t.commit_keys_per_thread = buckets, commit_keys
    hm = ash.HashMap(dim, 14_000_000, [(1,)], [torch.int32], tuning=t)  # a table of 224 MB
    n = 1_200_007
    g = torch.Generator(device="cuda").manual_seed(buckets + dim)
    v = torch.randint(0, n // 2, (n,), generator=g, device="cuda")
    keys = torch.stack([v * (j + 3) - 7 * j for j in range(dim)], 1).to(torch.int32).contiguous()
    first = torch.full((n // 2,), n, device="cuda", dtype=torch.int64)
    first.scatter_reduce_(0, v, torch.arange(n, device="cuda"), "amin")
    expect = first[v] == torch.arange(n, device="cuda")
    vals = torch.arange(n, device="cuda", dtype=torch.int32)[:, None].contiguous()
    idx, new = hm.insert(keys, [vals])
    assert torch.equal(new, expect) and torch.equal(idx >= 0, new)
    assert not hm.insert(keys, [vals + 1])[1].any()
    at, found = hm.find(keys)
    assert found.all() and torch.equal(hm.gather_values(at).view(-1).long(), first[v])
    assert hm.size() == int(expect.sum())
