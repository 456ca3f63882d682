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
