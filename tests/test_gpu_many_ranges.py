"""Calls partitioned into more than 32 home-bucket ranges (a table of several
gigabytes), at sizes around the partition's tiles: first occurrences win, and
every later call sees them."""
import pytest
import torch

from paper_2110_00511_gb300 import ash

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim", [1, 3, 8])
def test_partitioned_calls_on_a_large_table(dim):
    from paper_2110_00511_gb300 import build
    build.build()
    t = ash.default_tuning()
    t.partition_keys = 2
    hm = ash.HashMap(dim, 150_000_000 if dim == 8 else 290_000_000, tuning=t)
    assert hm.stats()["table_slots"] * 8 > 32 * (64 << 20)
    g = torch.Generator(device="cuda").manual_seed(dim)
    top = 0
    for n in (1, 31, 2047, 2049, 70_000, 1_234_567):
        v = top + torch.randint(0, max(1, n // 2), (n,), generator=g, device="cuda", dtype=torch.int32)
        top += max(1, n // 2)
        keys = torch.stack([v * (2 * j + 1) - j for j in range(dim)], 1).contiguous()
        first = torch.full((top,), n, device="cuda", dtype=torch.int64)
        first.scatter_reduce_(0, v.long(), torch.arange(n, device="cuda"), "amin")
        expect = first[v.long()] == torch.arange(n, device="cuda")
        idx, new = hm.activate(keys)
        assert torch.equal(new, expect)
        assert (idx[~new] == -1).all() and idx[new].unique().numel() == int(expect.sum())
        assert torch.equal(hm.gather_keys(idx[new]), keys[new])
        absent = keys.clone()
        absent[:, 0] = -absent[:, 0] - 1_000_000_000
        fidx, found = hm.find(torch.cat([keys, absent]).contiguous())
        assert found[:n].all() and not found[n:].any() and (fidx[n:] == -1).all()
        assert torch.equal(hm.gather_keys(fidx[:n]), keys)
        assert not hm.activate(keys)[1].any()
