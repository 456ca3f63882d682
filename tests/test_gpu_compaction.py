"""Ordered compaction on both sides of the tile counts that its write pass adds
up itself: the block keys of an image equal those of its two halves in turn,
and the double map's new keys are the winners of a plain activate, in order,
linked to the global entries."""
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


@pytest.mark.parametrize("width,height", [(1, 2), (511, 2), (256, 2), (19, 54), (1024, 2048), (1024, 2050), (2001, 1200)])
@pytest.mark.parametrize("sync", [True, False])
def test_depth_keys_keep_pixel_order(width, height, sync):
    g = torch.Generator(device="cuda").manual_seed(width)
    depth = torch.rand((height, width), generator=g, device="cuda") * 5
    depth[torch.rand((height, width), generator=g, device="cuda") < 0.3] = 0.0
    pose = torch.eye(3, 4)
    intr = (400.0, 410.0, width / 2, height // 2)

    def keys_of(image, cy):
        out = ash.ash_depth_to_block_keys(image.contiguous(), (*intr[:3], cy), pose, 0.05, 4.0, sync=sync)
        return out if sync else out[0][: int(out[1].item())]

    whole = keys_of(depth, float(intr[3]))
    half = height // 2
    parts = [keys_of(depth[:half], float(intr[3])), keys_of(depth[half:], float(intr[3] - half))]
    assert whole.shape[0] == int(((depth > 0) & (depth <= 4.0)).sum())
    assert torch.equal(whole, torch.cat(parts))


@pytest.mark.parametrize("n", [1, 512, 513, 2_097_152, 2_097_153])
@pytest.mark.parametrize("warp_probe", [0, 1])
def test_double_map_links_in_order(n, warp_probe):
    g = torch.Generator(device="cuda").manual_seed(n)
    keys = torch.randint(-20, 20, (n, 3), generator=g, device="cuda", dtype=torch.int32)
    t = ash.default_tuning()
    t.warp_probe = warp_probe
    local = ash.HashMap(3, n, [(1,)], [torch.int32])
    glob = ash.HashMap(3, 100_000, [(1,)], [torch.float32], tuning=t)
    glob.activate(keys[: n // 3].contiguous())
    mask = ash.HashMap(3, n).activate(keys)[1]
    unique, li, gi = ash.ash_double_map_activate(local, glob, keys)
    assert torch.equal(unique, keys[mask])
    assert torch.equal(local.find(unique)[0], li) and torch.equal(glob.find(unique)[0], gi) and (gi >= 0).all()
    assert torch.equal(local.gather_values(li).view(-1), gi)
