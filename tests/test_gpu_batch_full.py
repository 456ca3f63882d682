"""A batch of as many operations as one run takes (its descriptor table filled
to the last entry), against plain calls on twin maps; one more is refused."""
import pytest
import torch

from paper_2110_00511_gb300 import ash

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_ops", [1, 255, 256])
def test_a_batch_up_to_its_last_operation(n_ops):
    from paper_2110_00511_gb300 import build
    build.build()
    g = torch.Generator(device="cuda").manual_seed(n_ops)

    def keys(n):
        return torch.randint(-9, 9, (n, 3), generator=g, device="cuda", dtype=torch.int32)

    kinds = (ash.ASH_OP_INSERT, ash.ASH_OP_FIND, ash.ASH_OP_ERASE)
    maps = [[ash.HashMap(3, 1000, [(1,)], [torch.float32]) for _ in range(2)] for _ in range((n_ops + 2) // 3)]
    batch = ash.Batch()
    for _ in range(5):  # more rounds than the ring has slots
        items, plain = [], []
        for j in range(n_ops):
            batched, single = maps[j // 3]
            op, k = kinds[j % 3], keys(100 + j)
            val = torch.rand((len(k), 1), generator=g, device="cuda") if op == ash.ASH_OP_INSERT else None
            items.append((batched, op, k, val))
            plain.append(single.insert(k, [val])[1] if op == ash.ASH_OP_INSERT else
                         single.find(k)[1] if op == ash.ASH_OP_FIND else single.erase(k))
        for (_, mask), want in zip(batch.run(items), plain):
            assert torch.equal(mask, want)
    for batched, single in maps:
        probe = keys(3000)
        (a, found), (b, want) = batched.find(probe), single.find(probe)
        assert torch.equal(found, want) and torch.equal(batched.gather_values(a), single.gather_values(b))
        assert batched.size() == single.size()


def test_one_operation_too_many_is_refused():
    from paper_2110_00511_gb300 import build
    build.build()
    maps = [ash.HashMap(1, 16) for _ in range(257)]
    k = torch.zeros((1, 1), dtype=torch.int32, device="cuda")
    with pytest.raises(ash.AshError):
        ash.Batch().run([(m, ash.ASH_OP_FIND, k, None) for m in maps])
