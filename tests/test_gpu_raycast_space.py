"""Ray casting through much empty space: a plane far away whose blocks share
occupancy bits with nearer ones (the bits wrap every 128 blocks), partly full
4 x 4 x 4 cells, a map with freed indices, and voxel sizes on both sides of
the ones divided by multiplication (all lengths scaled by a power of two,
which scales every float32 step exactly)."""
import pytest
import torch

from paper_2110_00511_gb300 import ash

pytestmark = pytest.mark.gpu

EDGE = 8


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2110_00511_gb300 import build
    build.build()
    ash.lib()
    torch.cuda.init()


def plane_blocks(kz, voxel, z0, extra=()):
    """Blocks (x, y in -6..5, z in kz) holding the distance z0 - z at their lattice points, and `extra` blocks that hold
    free space (distance 1)."""
    xy = torch.arange(-6, 6, dtype=torch.int32, device="cuda")
    keys = torch.stack(torch.meshgrid(xy, xy, torch.tensor(kz, dtype=torch.int32, device="cuda"), indexing="ij"), -1).reshape(-1, 3)
    g = torch.arange(EDGE, device="cuda", dtype=torch.float32)
    z = (keys[:, 2].float()[:, None] * EDGE + g) * voxel  # [n, vz]
    d = (z0 - z)[:, :, None, None].expand(-1, EDGE, EDGE, EDGE)
    if len(extra):
        more = torch.tensor(extra, dtype=torch.int32, device="cuda")
        keys = torch.cat([keys, more])
        d = torch.cat([d, torch.ones((len(extra), EDGE, EDGE, EDGE), device="cuda")])
    return keys.contiguous(), d.contiguous()


@pytest.mark.parametrize("scale", [0, -54, -60, 40])
@pytest.mark.parametrize("through_local", [False, True])
@pytest.mark.parametrize("freed", [False, True])
@pytest.mark.parametrize("extra", [(), ((0, 0, 3), (1, -1, 3), (0, 0, 40), (-1, -1, 64), (200, 3, 1))])
@pytest.mark.parametrize("depth_min", [1, -3])
def test_a_far_plane_is_met_exactly(scale, through_local, freed, extra, depth_min):
    s = 2.0 ** scale
    voxel = s / 64
    z0 = (131 * EDGE + 3.5) * voxel
    keys, d = plane_blocks([131, 132], voxel, z0, extra)
    if scale < -50 or scale > 30:
        d = d / s  # distances need no scale of their own
    n = keys.shape[0]
    hm = ash.HashMap(3, 2 * n, [(EDGE,) * 3] * 2, [torch.float32] * 2)
    away = keys + torch.tensor([128, 256, -128], dtype=torch.int32, device="cuda")  # same occupancy bits
    hm.insert(away.contiguous(), [torch.ones_like(d), torch.zeros_like(d)])
    if freed:
        hm.erase(away[: n // 2].contiguous())
    hm.insert(keys, [d, torch.ones_like(d)])
    local = None
    if through_local:
        local = ash.HashMap(3, 2 * n, [(1,)], [torch.int32])
        idx, _ = hm.find(keys)
        local.insert(keys, [idx])
        if freed:
            local.erase(keys[n - 1:].contiguous())
    pose = torch.eye(3, 4)
    out = ash.ash_tsdf_raycast(hm, (200.0, 200.0, 7.5, 5.5), pose, 17, 13, voxel, depth_min * voxel, voxel, 140 * EDGE,
                               local=local)
    # samples lie on the lattice in z, so a linear distance is met where it is zero
    assert torch.equal(out, torch.full_like(out, z0)), (out / z0).unique()
