"""Keys that come in runs of equal ones (scan order), across warp and block
edges: the first occurrence wins, in every claim protocol and with points."""
import pytest
import torch

from paper_2110_00511_gb300 import ash

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("run", [1, 2, 31, 32, 33, 300])
@pytest.mark.parametrize("n", [1, 33, 10_007])
@pytest.mark.parametrize("dim,claim_mode", [(1, 2), (3, 2), (3, 1), (4, 0), (8, 2)])
def test_runs_of_equal_keys(run, n, dim, claim_mode):
    from paper_2110_00511_gb300 import build
    build.build()
    t = ash.default_tuning()
    t.claim_mode = claim_mode
    v = torch.arange(n, device="cuda", dtype=torch.int32) // run % 50  # each run comes back later
    keys = torch.stack([v * (j + 1) - j for j in range(dim)], 1).contiguous()
    first = torch.full((50,), n, device="cuda", dtype=torch.int64)
    first.scatter_reduce_(0, v.long(), torch.arange(n, device="cuda"), "amin")
    expect = first[v.long()] == torch.arange(n, device="cuda")
    vals = torch.arange(n, device="cuda", dtype=torch.int32)[:, None].contiguous()
    for points in (False, True):
        hm = ash.HashMap(dim, n, [(1,)], [torch.int32], tuning=t)
        for again in (False, True):
            idx, new = hm.insert_points(keys.float() + 0.5, 1.0, [vals]) if points else hm.insert(keys, [vals])
            assert torch.equal(new, expect & (not again)) and torch.equal(idx >= 0, new)
        assert torch.equal(hm.gather_values(hm.find(keys)[0]).view(-1).long(), first[v.long()])
