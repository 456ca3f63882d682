"""Value rows written by insert, read by gather_values and moved by a
compacting rehash, at every element width (16, 8, 4, 2, 1 bytes), odd row
sizes and ragged counts: byte-exact against plain indexing."""
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


@pytest.mark.parametrize("row_bytes", [1, 2, 3, 4, 6, 8, 10, 12, 16, 24, 33, 512, 2048])
@pytest.mark.parametrize("n", [1, 31, 1025, 70_001])
def test_value_rows(row_bytes, n):
    if row_bytes * n > 1 << 25:
        n = (1 << 25) // row_bytes
    g = torch.Generator(device="cuda").manual_seed(row_bytes * 1000 + n)
    distinct = torch.arange(n, dtype=torch.int32, device="cuda") * 7 - 3
    keys = torch.stack([distinct, -distinct], 1).contiguous()
    twice = torch.cat([keys, keys.flip(0)]).contiguous()  # the second occurrence of each key loses
    vals = torch.randint(0, 256, (2 * n, row_bytes), generator=g, device="cuda", dtype=torch.int32).to(torch.uint8)
    other = vals.flip(1).contiguous()
    hm = ash.HashMap(2, 4 * n, [(row_bytes,), (row_bytes,)], [torch.uint8] * 2)
    hm.insert(twice, [vals, other])
    for capacity in (None, n):  # as inserted, then compacted
        if capacity:
            hm.erase(keys[: n // 2].contiguous())
            hm.rehash(capacity)
        idx, mask = hm.find(keys)
        assert mask.sum().item() == (n if capacity is None else n - n // 2)
        expect = torch.where(mask[:, None], vals[:n], torch.zeros_like(vals[:n]))
        assert torch.equal(hm.gather_values(idx, 0), expect)
        assert torch.equal(hm.gather_values(idx, 1), expect.flip(1))
        bad = torch.tensor([-1, hm.capacity(), idx.max().item(), 2**31 - 1], dtype=torch.int32, device="cuda")
        rows = hm.gather_values(bad, 0)
        assert not rows[[0, 1, 3]].any()
        assert torch.equal(rows[2], hm.value_buffer(0)[idx.max().item()])
        unaligned = torch.empty(row_bytes * n + 1, dtype=torch.uint8, device="cuda")[1:]
        ash._check(ash.lib().ash_gather_values(hm.handle, 0, idx.data_ptr(), n, unaligned.data_ptr(), ash._stream()))
        assert torch.equal(unaligned.view(n, row_bytes), expect)


@pytest.mark.parametrize("row_bytes", [1, 3, 10, 16, 100])
@pytest.mark.parametrize("capacity,grown", [(1, 2), (7, 29), (1001, 70_003)])
@pytest.mark.parametrize("erased", [False, True])
@pytest.mark.parametrize("how", ["rehash", "reserve_async", "insert", "shrink"])
def test_storage_moves_keep_entries(row_bytes, capacity, grown, erased, how):
    """Growth (with the count known to the host or only to the device) and
    compaction, with and without freed indices before them: indices, rows and
    heap kept, new value rows zero, and the map usable to its new capacity."""
    g = torch.Generator(device="cuda").manual_seed(capacity + row_bytes)
    k = torch.arange(grown, dtype=torch.int32, device="cuda")
    keys = torch.stack([k, -3 * k, k ^ 5], 1).contiguous()
    vals = torch.randint(0, 256, (grown, row_bytes), generator=g, device="cuda", dtype=torch.int32).to(torch.uint8)
    hm = ash.HashMap(3, grown if how == "shrink" else capacity, [(row_bytes,)], [torch.uint8])
    hm.insert(keys[:capacity].contiguous(), [vals[:capacity].contiguous()])
    kept = torch.ones(capacity, dtype=torch.bool, device="cuda")
    if erased:
        kept[::2] = False
        hm.erase(keys[:capacity][::2].contiguous())
    before, _ = hm.find(keys[:capacity].contiguous())
    if how == "rehash":
        hm.rehash(grown)
    elif how == "reserve_async":
        hm.reserve_async(grown)
    elif how == "shrink":
        hm.rehash(capacity)
    else:
        hm.insert(keys[capacity:].contiguous(), [vals[capacity:].contiguous()])
    idx, mask = hm.find(keys[:capacity].contiguous())
    assert torch.equal(mask, kept)
    if how != "shrink":
        assert torch.equal(idx, before)
    assert torch.equal(hm.gather_values(idx), torch.where(kept[:, None], vals[:capacity], torch.zeros_like(vals[:capacity])))
    live = capacity - (capacity + 1) // 2 if erased else capacity
    live += grown - capacity if how == "insert" else 0
    stats = hm.stats()
    assert (stats["live"], stats["used_slots"]) == (live, live) or how == "insert"
    assert hm.size() == live and hm.active_indices().unique().numel() == live
    h, t = hm.heap()
    assert t == live
    assert torch.equal(torch.cat([hm.active_indices(), h[t:]]).sort().values,
                       torch.arange(hm.capacity(), dtype=torch.int32, device="cuda"))
    if how in ("rehash", "reserve_async"):
        assert not hm.value_buffer(0)[capacity:].any()
    fill = min(grown, hm.capacity())
    hm.insert(keys[:fill].contiguous(), [vals[:fill].contiguous()])
    hm.sync_status()
    idx, mask = hm.find(keys[:fill].contiguous())
    assert mask.all() and torch.equal(hm.gather_values(idx), vals[:fill])
    hm.clear()
    assert hm.size() == 0 and not hm.find(keys)[1].any()
    assert torch.equal(hm.heap()[0], torch.arange(hm.capacity(), dtype=torch.int32, device="cuda"))
