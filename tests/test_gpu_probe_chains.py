"""Lookups whose probe chains run past the home bucket: tables filled close to
their slots, every bucket size and keys per thread, against the positions the
keys were inserted at; and the neighbour queries over such tables against the
materialised ones, at every radius (the offset numbers' division)."""
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


def dense_map(n, dim, buckets, keys_per_thread=1, seed=0):
    """A map filled to 1 / 1.05 of its slots: (map, its n keys, the value of each)."""
    t = ash.default_tuning()
    t.slots_per_bucket, t.slots_per_capacity, t.max_used_fraction = buckets, 1.05, 0.98
    t.find_keys_per_thread = keys_per_thread
    g = torch.Generator(device="cuda").manual_seed(seed)
    side = max(2, round(n ** (1 / dim)) + 1)
    keys = torch.stack([torch.arange(n, device="cuda", dtype=torch.int32) // side ** j % side if j < dim - 1
                        else torch.arange(n, device="cuda", dtype=torch.int32) // side ** j for j in range(dim)], 1)
    keys = keys[torch.randperm(n, generator=g, device="cuda")].contiguous()
    hm = ash.HashMap(dim, n, [(1,)], [torch.int32], tuning=t)
    hm.insert(keys, [torch.arange(n, device="cuda", dtype=torch.int32)])
    hm.sync_status()
    return hm, keys


@pytest.mark.parametrize("buckets", [4, 8, 16])
@pytest.mark.parametrize("keys_per_thread", [1, 2, 4])
@pytest.mark.parametrize("n,dim", [(5, 1), (257, 2), (40_001, 3), (3_000, 8)])
def test_find_past_the_home_bucket(buckets, keys_per_thread, n, dim):
    hm, keys = dense_map(n, dim, buckets, keys_per_thread)
    absent = keys.clone()
    absent[:, 0] += 1 << 20
    queries = torch.cat([keys, absent]).contiguous()
    idx, mask = hm.find(queries)
    assert mask[:n].all() and not mask[n:].any() and (idx[n:] == -1).all()
    assert torch.equal(hm.gather_values(idx[:n]).view(-1), torch.arange(n, device="cuda", dtype=torch.int32))
    t = hm.tuning()
    t.max_probes = 1  # only the home bucket: what is found is right, and nothing past it is
    hm.set_tuning(t)
    idx1, mask1 = hm.find(queries)
    assert torch.equal(idx1[mask1], idx[mask1]) and not mask1[n:].any()
    assert mask1[:n].float().mean() < 1 or n < 16


@pytest.mark.parametrize("dim,radius", [(1, 0), (1, 8), (2, 1), (2, 5), (3, 0), (3, 1), (3, 3), (4, 2), (5, 1)])
@pytest.mark.parametrize("buckets", [4, 16])
def test_neighbors_past_the_home_bucket(dim, radius, buckets):
    hm, keys = dense_map(1_501, dim, buckets)
    q = keys[:333].contiguous()
    span = torch.arange(-radius, radius + 1, device="cuda", dtype=torch.int32)
    off = torch.stack(torch.meshgrid(*[span] * dim, indexing="ij"), -1).reshape(-1, dim).contiguous()
    want, want_mask = hm.find((q[:, None] + off[None]).reshape(-1, dim).contiguous())
    idx, mask = hm.find_neighbors(q, radius)
    assert torch.equal(idx.view(-1), want) and torch.equal(mask.view(-1), want_mask)
    if off.shape[0] <= 4096:
        idx, mask = hm.find_offsets(q, off)
        assert torch.equal(idx.view(-1), want) and torch.equal(mask.view(-1), want_mask)
