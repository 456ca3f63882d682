"""The work that programs built on this package give it, as cases to be timed.

Every case is one pass of such a program through the package's public entry
points: calls on hash sets and maps (small, ordinary and larger than L2),
voxelization of point clouds, a sliding window of keys, many maps in one
batched launch, growth from a small capacity, neighbour tables, checkpoints,
and the voxel-block pipeline (one frame of TSDF fusion, one rendered view).

Buffer indices are handed out in the order in which the GPU's blocks reach the
index heap, so two runs on the same inputs number their entries differently.
A pass therefore returns the masks and what a program reads through the
indices (the value rows), which the inputs alone determine.
"""
from __future__ import annotations

import math

import torch

from paper_2110_00511_gb300 import ash

DTYPES = {"f32": torch.float32, "f16": torch.float16, "i32": torch.int32, "f64": torch.float64, "u8": torch.uint8}
SPAN = 1 << 20  # uniform key coordinates lie in [-SPAN, SPAN)


def listed():
    return [
        # one small query against a map that is already there (a picked region, one scan line): latency
        {"name": "lookup_4k", "kind": "lookup", "entries": 200_000, "n": 4_096, "dim": 3, "dtype": "f32", "numel": 1,
         "hits": 0.5},
        # a per-scan hash set of ten thousand keys: clear, activate, find
        {"name": "set_10k", "kind": "set", "n": 10_000, "dim": 3, "rho": 0.5},
        # the uniqueness sweep's largest size: a table twelve times the L2 cache
        {"name": "set_100m", "kind": "set", "n": 100_000_000, "dim": 3, "rho": 0.5},
        # bulk lookups of feature rows on a 4-D grid, half of the queries absent
        {"name": "lookup_6m_4d", "kind": "lookup", "entries": 5_000_000, "n": 6_000_001, "dim": 4, "dtype": "f16",
         "numel": 8, "hits": 0.5},
        # voxelization of a point cloud at 5 mm, nearly all voxels distinct: the benchmark's step
        {"name": "voxelize_4m_5mm", "kind": "voxelize", "n": 4_000_000, "voxel": 0.005, "fused": False},
        # a smaller scan at 50 mm: several points per voxel, a ragged point count, quantised inside the hash kernels
        {"name": "voxelize_1m_50mm", "kind": "voxelize", "n": 1_000_003, "voxel": 0.05, "fused": True},
        # a sliding window: each pass brings a batch of keys, looks keys up and drops the batch again
        {"name": "window_1m", "kind": "window", "entries": 1_000_000, "batch": 262_145, "n": 500_000, "dim": 3,
         "dtype": "f32", "numel": 4},
        # 24 tenants' maps in one batched launch, insert / find / erase for each
        {"name": "batch_24_maps", "kind": "batch", "maps": 24, "log2_lo": 10.0, "log2_hi": 20.0},
        # a map whose size nobody knew: chunks inserted from a small capacity, doubling on the way
        {"name": "grow_1m", "kind": "grow", "start": 16_384, "chunk": 100_000, "chunks": 12, "dim": 3},
        # the 27-neighbourhood of every surface block of a scene, and what it holds
        {"name": "neighbors_200k", "kind": "neighbors", "n": 200_000, "dim": 3, "table": "radius"},
        # a checkpoint of a block map (8^3 rows in two types), loaded again
        {"name": "checkpoint_40k", "kind": "checkpoint", "n": 40_000, "dim": 3, "ell": 8},
        # one depth frame fused into the volume and the surface seen again: a whole call of the block pipeline
        {"name": "fuse_frame_vga", "kind": "frame", "width": 640, "height": 480, "voxel": 0.006, "ell": 8, "size": 4.0},
    ]


def draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["lookup", "lookup", "set", "set", "voxelize", "voxelize", "window", "window", "batch", "grow",
                       "neighbors", "checkpoint", "frame"])
    if kind == "lookup":
        dtype, numel = rng.choice([("f32", 1), ("f16", 8), ("f32", 3), ("f64", 1), ("u8", 3), ("f32", 32), ("i32", 2)])
        return {"kind": kind, "entries": log(10_000, 5_000_000), "n": log(1_000, 6_000_000), "dim": rng.randint(2, 8),
                "dtype": dtype, "numel": numel, "hits": round(rng.uniform(0.1, 0.95), 2)}
    if kind == "set":
        return {"kind": kind, "n": log(5_000, 90_000_000), "dim": rng.randint(2, 5), "rho": round(rng.uniform(0.1, 1), 2)}
    if kind == "voxelize":
        return {"kind": kind, "n": log(100_000, 4_000_000), "voxel": rng.choice([0.005, 0.01, 0.02, 0.05]),
                "fused": rng.random() < 0.5}
    if kind == "window":
        dtype, numel = rng.choice([("f32", 1), ("f32", 4), ("f64", 1), ("f16", 5), ("f32", 16)])
        entries = log(50_000, 4_000_000)
        return {"kind": kind, "entries": entries, "batch": max(1_000, int(entries * rng.uniform(0.2, 0.4))),
                "n": log(10_000, 2_000_000), "dim": rng.randint(2, 4), "dtype": dtype, "numel": numel}
    if kind == "batch":
        return {"kind": kind, "maps": rng.randint(4, 48), "log2_lo": 10.0, "log2_hi": round(rng.uniform(14, 21), 2)}
    if kind == "grow":
        return {"kind": kind, "start": 1 << rng.randint(10, 16), "chunk": log(10_000, 300_000),
                "chunks": rng.randint(4, 16), "dim": rng.randint(2, 4)}
    if kind == "neighbors":
        dim = rng.randint(2, 4)
        return {"kind": kind, "n": log(10_000, 150_000), "dim": dim, "table": rng.choice(["radius", "cube", "ring"])}
    if kind == "checkpoint":
        ell = rng.choice([1, 2, 4, 8])
        return {"kind": kind, "n": log(10_000, 400_000 if ell < 8 else 50_000), "dim": 3, "ell": ell}
    w = rng.randrange(200, 640)
    return {"kind": kind, "width": w, "height": w * 3 // 4, "voxel": rng.choice([0.006, 0.008, 0.01]),
            "ell": rng.choice([8, 16]), "size": round(rng.uniform(3.0, 5.0), 2)}


# ------------------------------------------------------------------- inputs
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _ints(g, lo, hi, *shape):
    return torch.randint(lo, hi, shape, generator=g, device="cuda", dtype=torch.int32)


def _uniform_keys(g, n, dim, shift=0):
    """n uniform rows, the first coordinate moved by `shift` (disjoint ranges)."""
    k = _ints(g, -SPAN, SPAN, n, dim)
    if shift:
        k[:, 0] += shift
    return k


def _pick(g, rows, n):
    return rows[torch.randint(0, rows.shape[0], (n,), generator=g, device="cuda")]


def _shuffled(g, rows):
    return rows[torch.randperm(rows.shape[0], generator=g, device="cuda")].contiguous()


def _rho_keys(g, n, dim, rho):
    """n rows with about rho * n distinct keys, in random order."""
    u = max(1, min(n, round(rho * n)))
    distinct = _uniform_keys(g, u, dim)
    return _shuffled(g, torch.cat([distinct, _pick(g, distinct, n - u)])) if u < n else distinct


def _values(g, n, dtype, numel):
    if dtype in ("i32", "u8"):
        return torch.randint(0, 256, (n, numel), generator=g, device="cuda", dtype=torch.int32).to(DTYPES[dtype])
    return torch.randn((n, numel), generator=g, device="cuda").to(DTYPES[dtype])


def _scene_points(g, n, room=10.0, n_spheres=32, noise=0.002):
    """float32 [n, 3] points on spheres and the three walls of a room, by area, with sensor noise, in random order."""
    centre = torch.rand((n_spheres, 3), generator=g, device="cuda") * room
    radius = 0.2 + 1.3 * torch.rand(n_spheres, generator=g, device="cuda")
    area = torch.cat([4 * math.pi * radius ** 2, torch.full((3,), room * room, device="cuda")])
    on = torch.multinomial(area, n, replacement=True, generator=g)
    d = torch.randn((n, 3), generator=g, device="cuda")
    d /= d.norm(dim=1, keepdim=True)
    s = on.clamp(max=n_spheres - 1)
    p = centre[s] + radius[s, None] * d
    flat = torch.rand((n, 3), generator=g, device="cuda") * room
    flat.scatter_(1, (on - n_spheres).clamp(min=0)[:, None], 0.0)
    p = torch.where((on >= n_spheres)[:, None], flat, p)
    return (p + noise * torch.randn((n, 3), generator=g, device="cuda")).contiguous()


def _surface_keys(g, n, dim):
    """n distinct cell keys on the surfaces of a scene: axis-aligned faces swept cell by cell, as a scan meets them, with
    a tenth of the cells unseen."""
    want, n = n, n + n // 9
    side = max(2, math.ceil((n / 6) ** (1.0 / max(1, dim - 1))) + 1)
    span = torch.arange(side, device="cuda", dtype=torch.int32)
    faces = []
    for f in range(6):
        axis = f % dim
        grid = torch.stack(torch.meshgrid(*[span] * (dim - 1), indexing="ij"), -1).reshape(-1, dim - 1)
        fixed = torch.full((grid.shape[0], 1), (f // dim + 1) * 3 * side, device="cuda", dtype=torch.int32)
        faces.append(torch.cat([grid[:, :axis], fixed, grid[:, axis:]], 1))
    keys = torch.cat(faces)
    while keys.shape[0] < n:  # few cells per face (2-D): more faces further away
        keys = torch.cat([keys, keys + 7 * side])
    seen = torch.randperm(n, generator=g, device="cuda")[:want].sort().values
    return (keys[seen] + _ints(g, -500, 500, 1, dim)).contiguous()


# ------------------------------------------------- room, camera (voxel blocks)
def _pose(angle, size):
    """World-to-camera [R | t] rows of a level camera near the room's centre, looking along `angle`."""
    c, s = math.cos(angle), math.sin(angle)
    r = torch.tensor([[s, -c, 0.0], [0.0, 0.0, -1.0], [c, s, 0.0]], dtype=torch.float64)
    pos = torch.tensor([size / 2 + 0.3 * s, size / 2 - 0.3 * c, size * 0.4], dtype=torch.float64)
    return torch.cat([r, -(r @ pos)[:, None]], 1).float()


def _camera(case):
    f = 525.0 * case["width"] / 640.0
    return (f, f, (case["width"] - 1) / 2, (case["height"] - 1) / 2)


def _room_depth(g, case, pose, spheres):
    """float32 [H, W] depth of a closed room with spheres inside, with sensor noise and a few missing pixels."""
    h, w, size = case["height"], case["width"], case["size"]
    fx, fy, cx, cy = _camera(case)
    e = pose.double().cuda()
    r, pos = e[:, :3], -(e[:, :3].T @ e[:, 3])
    v, u = torch.meshgrid(torch.arange(h, device="cuda", dtype=torch.float64),
                          torch.arange(w, device="cuda", dtype=torch.float64), indexing="ij")
    d = torch.stack([(u - cx) / fx, (v - cy) / fy, torch.ones_like(u)], -1) @ r
    best = torch.full((h, w), 1e9, device="cuda", dtype=torch.float64)
    for axis in range(3):
        for wall in (0.0, size):
            t = (wall - pos[axis]) / d[..., axis]
            best = torch.where((t > 0) & (t < best), t, best)
    a = (d * d).sum(-1)
    for k in range(spheres.shape[0]):
        oc = pos - spheres[k, :3]
        b = 2 * (d @ oc)
        disc = b * b - 4 * a * ((oc * oc).sum() - spheres[k, 3] ** 2)
        t = (-b - disc.clamp(min=0).sqrt()) / (2 * a)
        best = torch.where((disc > 0) & (t > 0) & (t < best), t, best)
    depth = best.float() + 0.002 * torch.randn((h, w), generator=g, device="cuda")
    return torch.where(torch.rand((h, w), generator=g, device="cuda") < 0.01, torch.zeros_like(depth), depth).contiguous()


def _frames(case, seed):
    """The frame to fuse and the ones before it: [(depth, pose)], the last one new."""
    g = _gen(seed)
    size = case["size"]
    spheres = torch.cat([0.4 + (size - 0.8) * torch.rand((8, 3), generator=g, device="cuda"),
                         0.1 + 0.25 * torch.rand((8, 1), generator=g, device="cuda")], 1).double()
    start = 6.0 * torch.rand(1, generator=g, device="cuda").item()
    poses = [_pose(start + 0.06 * j, size) for j in range(4)]
    return [(_room_depth(g, case, p, spheres), p) for p in poses]


def _frame_rows(case):
    """Block rows of a frame's output buffers: a good part of the blocks of one wall of the room."""
    return int(0.4 * (case["size"] / (case["voxel"] * case["ell"])) ** 2)


def _ray(case):
    """depth_min, step and sample count of the ray caster, and the depth limit of the sensor."""
    limit = 2.0 * case["size"]
    step = 0.75 * case["voxel"]
    return 0.2, step, int((limit - 0.2) / step), limit


def _fuse(case, state, depth, pose):
    """One frame of the block pipeline: the frame's blocks, allocation in both maps, integration."""
    intr, voxel = _camera(case), case["voxel"]
    limit = _ray(case)[3]
    state["local"].clear()
    keys = ash.ash_depth_to_block_keys(depth, intr, pose, voxel * case["ell"], limit)
    unique, _, index = ash.ash_double_map_activate(state["local"], state["blocks"], keys)
    ash.ash_tsdf_integrate(state["blocks"], index, depth, intr, pose, voxel, 4 * voxel, limit)
    return unique, index


# ----------------------------------------------------------------- prepare
def prepare(case, seed):
    g = _gen(seed)
    kind = case["kind"]
    if kind == "lookup":
        keys = _uniform_keys(g, case["entries"], case["dim"])
        hm = ash.HashMap(case["dim"], case["entries"], [(case["numel"],)], [DTYPES[case["dtype"]]])
        hm.insert(keys, [_values(g, case["entries"], case["dtype"], case["numel"])])
        hit = int(case["n"] * case["hits"])
        absent = _uniform_keys(g, case["n"] - hit, case["dim"], shift=4 * SPAN)
        return {"case": case, "map": hm, "queries": _shuffled(g, torch.cat([_pick(g, keys, hit), absent]))}
    if kind == "set":
        keys = _rho_keys(g, case["n"], case["dim"], case["rho"])
        half = case["n"] // 2
        other = torch.cat([keys[:half], _uniform_keys(g, case["n"] - half, case["dim"], shift=4 * SPAN)])
        return {"case": case, "map": ash.HashMap(case["dim"], case["n"]), "keys": keys, "queries": _shuffled(g, other)}
    if kind == "voxelize":
        return {"case": case, "points": _scene_points(g, case["n"]),
                "ids": torch.arange(case["n"], dtype=torch.int32, device="cuda")}
    if kind == "window":
        dim, numel, dtype = case["dim"], case["numel"], case["dtype"]
        base = _uniform_keys(g, case["entries"], dim)
        hm = ash.HashMap(dim, 2 * case["entries"], [(numel,)], [DTYPES[dtype]])
        hm.insert(base, [_values(g, case["entries"], dtype, numel)])
        third = case["n"] // 3
        steps = []
        for _ in range(4):  # the batches that come and go, one per pass
            fresh = _uniform_keys(g, case["batch"], dim, shift=4 * SPAN)
            queries = torch.cat([_pick(g, base, third), _pick(g, fresh, third),
                                 _uniform_keys(g, case["n"] - 2 * third, dim, shift=8 * SPAN)])
            steps.append((fresh, _values(g, case["batch"], dtype, numel), _shuffled(g, queries)))
        return {"case": case, "map": hm, "steps": steps, "turn": 0}
    if kind == "batch":
        sizes = _batch_sizes(case, seed)
        items = []
        for dim, cap in sizes:
            hm = ash.HashMap(dim, cap, [(1,)], [torch.float32])
            base = _uniform_keys(g, cap // 2, dim)
            hm.insert(base, [_values(g, cap // 2, "f32", 1)])
            fresh = _uniform_keys(g, max(1, cap // 8), dim, shift=4 * SPAN)
            half = max(1, cap // 8)
            queries = torch.cat([_pick(g, base, half), _pick(g, fresh, half),
                                 _uniform_keys(g, half, dim, shift=8 * SPAN)])
            items += [(hm, ash.ASH_OP_INSERT, fresh, _values(g, fresh.shape[0], "f32", 1)),
                      (hm, ash.ASH_OP_FIND, _shuffled(g, queries), None), (hm, ash.ASH_OP_ERASE, fresh, None)]
        # outputs in two arenas that the program keeps
        counts = [keys.shape[0] for _, _, keys, _ in items]
        index = torch.empty(sum(counts), dtype=torch.int32, device="cuda").split(counts)
        masks = torch.empty(sum(counts), dtype=torch.bool, device="cuda")
        outputs = [(i if item[1] != ash.ASH_OP_ERASE else None, m) for item, i, m in zip(items, index, masks.split(counts))]
        return {"case": case, "batch": ash.Batch(), "items": items, "outputs": outputs, "masks": masks}
    if kind == "grow":
        n = case["chunk"] * case["chunks"]
        keys = _rho_keys(g, n, case["dim"], 0.8)
        return {"case": case, "chunks": list(keys.split(case["chunk"])),
                "values": list(_values(g, n, "f32", 1).split(case["chunk"])), "queries": _shuffled(g, keys)}
    if kind == "neighbors":
        keys = _surface_keys(g, case["n"], case["dim"])
        hm = ash.HashMap(case["dim"], case["n"], [(1,)], [torch.int32])
        hm.insert(keys, [_ints(g, 0, 1 << 30, case["n"], 1)])
        return {"case": case, "map": hm, "keys": keys, "offsets": _offsets(case)}
    if kind == "checkpoint":
        n, ell = case["n"], case["ell"]
        keys = _surface_keys(g, n, case["dim"])
        shape = (ell, ell, ell)
        hm = ash.HashMap(case["dim"], n + n // 2, [shape, shape], [torch.float32, torch.float16])
        rows = torch.randn((n, *shape), generator=g, device="cuda")
        hm.insert(keys, [rows, rows.half()])
        return {"case": case, "map": hm, "queries": _pick(g, keys, n // 4)}
    cells = int(case["size"] / (case["voxel"] * case["ell"])) + 3
    state = {"case": case, "frames": _frames(case, seed), "local": ash.HashMap(3, 1 << 19, [(1,)], [torch.int32]),
             "blocks": ash.HashMap(3, 12 * cells * cells, [(case["ell"],) * 3] * 2, [torch.float32] * 2)}
    for depth, pose in state["frames"][:-1]:
        _fuse(case, state, depth, pose)
    return state


def _batch_sizes(case, seed):
    """(key dimension, capacity) of each map: dimensions 2..4, capacities spread evenly over the logarithm."""
    m = case["maps"]
    caps = [int(2 ** (case["log2_lo"] + (case["log2_hi"] - case["log2_lo"]) * (j + 0.5) / m)) for j in range(m)]
    return [(2 + (j * 7) % 3, caps[(j * 5) % m] if m % 5 else caps[j]) for j in range(m)]


def _offsets(case):
    """The neighbour table of the case: the 3^d radius, the 2^d cube or the 2d ring."""
    dim = case["dim"]
    if case["table"] == "ring":
        eye = torch.eye(dim, dtype=torch.int32, device="cuda")
        return torch.cat([-eye, eye]).contiguous()
    span = torch.arange(2, dtype=torch.int32, device="cuda")
    return torch.stack(torch.meshgrid(*[span] * dim, indexing="ij"), -1).reshape(-1, dim).contiguous()


# --------------------------------------------------------------------- run
def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "lookup":
        index, mask = state["map"].find(state["queries"])
        return {"mask": mask, "values": state["map"].gather_values(index)}
    if kind == "set":
        hm = state["map"]
        hm.clear()
        _, new = hm.activate(state["keys"])
        _, found = hm.find(state["queries"])
        return {"new": new, "found": found}
    if kind == "voxelize":
        points, n = state["points"], case["n"]
        hm = ash.HashMap(3, n, [(1,)], [torch.int32])
        if case["fused"]:
            _, first = hm.insert_points(points, case["voxel"], [state["ids"]])
            index, mask = hm.find_points(points, case["voxel"])
            return {"first": first, "mask": mask, "voxel_of_point": hm.gather_values(index)}
        keys = ash.ash_quantize(points, case["voxel"])
        _, first = hm.insert(keys, [state["ids"]])
        index, mask = hm.find(keys)
        return {"keys": keys, "first": first, "mask": mask, "voxel_of_point": hm.gather_values(index)}
    if kind == "window":
        hm = state["map"]
        fresh, rows, queries = state["steps"][state["turn"] % len(state["steps"])]
        state["turn"] += 1
        _, new = hm.insert(fresh, [rows])
        index, found = hm.find(queries)
        values = hm.gather_values(index)
        return {"new": new, "found": found, "values": values, "erased": hm.erase(fresh)}
    if kind == "batch":
        state["batch"].run(state["items"], outputs=state["outputs"])
        return {"masks": state["masks"]}
    if kind == "grow":
        hm = ash.HashMap(case["dim"], case["start"], [(1,)], [torch.float32])
        new = [hm.insert(k, [v])[1] for k, v in zip(state["chunks"], state["values"])]
        index, found = hm.find(state["queries"])
        return {"new": new, "found": found, "values": hm.gather_values(index)}
    if kind == "neighbors":
        hm = state["map"]
        if case["table"] == "radius":
            index, mask = hm.find_neighbors(state["keys"], 1)
        else:
            index, mask = hm.find_offsets(state["keys"], state["offsets"])
        return {"mask": mask, "ids": hm.gather_values(index.view(-1))}
    if kind == "checkpoint":
        copy = ash.HashMap.from_export(state["map"].export())
        index, found = copy.find(state["queries"])
        return {"found": found, "f32": copy.gather_values(index, 0), "f16": copy.gather_values(index, 1)}
    depth, pose = state["frames"][-1]
    unique, index = _fuse(case, state, depth, pose)
    depth_min, step, n_steps, _ = _ray(case)
    blocks = state["blocks"]
    # handed to the mesher in buffers of a fixed size: -1 (a zero row) where the frame has fewer blocks
    rows = torch.full((_frame_rows(case),), -1, dtype=torch.int32, device="cuda")
    keys = torch.zeros((rows.shape[0], 3), dtype=torch.int32, device="cuda")
    u = min(index.shape[0], rows.shape[0])
    rows[:u] = index[:u]
    keys[:u] = unique[:u]
    seen = ash.ash_tsdf_raycast(blocks, _camera(case), pose, case["width"], case["height"], case["voxel"], depth_min,
                                step, n_steps, local=state["local"])
    return {"blocks": keys, "tsdf": blocks.gather_values(rows, 0), "weight": blocks.gather_values(rows, 1),
            "seen": seen}


# -------------------------------------------------------------------- work
def work(case):
    """Bytes: inputs and outputs once, and of the map the slots (8 bytes), key rows and value rows touched; flops: the
    voxel updates of a fused frame, and nothing worth counting elsewhere."""
    kind = case["kind"]
    if kind == "lookup":
        row = case["numel"] * DTYPES[case["dtype"]].itemsize
        n, hit = case["n"], int(case["n"] * case["hits"])
        return {"bytes": n * (4 * case["dim"] + 8 + 5 + 4 + row) + hit * (4 * case["dim"] + row), "flops": 0}
    if kind == "set":
        n, u, key = case["n"], int(case["n"] * case["rho"]), 4 * case["dim"]
        table = 16 * n  # cleared: every slot written
        return {"bytes": table + n * (key + 8 + 5) + u * (key + 8) + n * (key + 8 + 5) + n // 2 * key, "flops": 0}
    if kind == "voxelize":
        n = case["n"]
        quantised = 0 if case["fused"] else 12 * n
        # the table and the values initialised; per point its row twice, slots, outputs, the voxel's row
        return {"bytes": 16 * n + 4 * n + quantised + n * (12 + 8 + 5) + n * (12 + 4 + 8)
                + n * (12 + 8 + 12 + 5) + n * (4 + 4 + 4), "flops": 0}
    if kind == "window":
        row = case["numel"] * DTYPES[case["dtype"]].itemsize
        key, b, n = 4 * case["dim"], case["batch"], case["n"]
        insert = b * (key + 8 + 5 + key + row + row + 8)
        find = n * (key + 8 + 5 + 4 + row) + 2 * (n // 3) * (key + row)
        return {"bytes": insert + find + b * (key + 8 + key + 8 + 4 + 1), "flops": 0}
    if kind == "batch":
        total = 0
        for dim, cap in _batch_sizes(case, 0):
            key, b, n = 4 * dim, max(1, cap // 8), 3 * max(1, cap // 8)
            total += b * (key + 8 + 5 + key + 4 + 4 + 8) + n * (key + 8 + 5) + 2 * n // 3 * key
            total += b * (key + 8 + key + 8 + 4 + 1)
        return {"bytes": total, "flops": 0}
    if kind == "grow":
        n, key = case["chunk"] * case["chunks"], 4 * case["dim"]
        u = int(0.8 * n)
        final = case["start"]
        while final < u:
            final *= 2
        return {"bytes": 16 * final + 4 * final + n * (key + 8 + 5 + 4) + u * (key + 4 + 8)
                + n * (key + 8 + key + 5 + 4 + 4 + 4), "flops": 0}
    if kind == "neighbors":
        n, dim = case["n"], case["dim"]
        offsets = {"radius": 3 ** dim, "cube": 2 ** dim, "ring": 2 * dim}[case["table"]]
        hits = n * offsets // 3
        return {"bytes": n * 4 * dim + n * offsets * (8 + 5 + 4 + 4) + hits * (4 * dim + 4), "flops": 0}
    if kind == "checkpoint":
        n, key, row = case["n"], 4 * case["dim"], 6 * case["ell"] ** 3
        cap = n + n // 2
        read = n * (4 + key + row)
        # the copy's table and value buffers initialised, its rows written; a quarter of the rows read back
        return {"bytes": 2 * read + 16 * cap + cap * row + n * (key + row + 8) + n // 4 * (key + 8 + key + 5 + 2 * row),
                "flops": 0}
    pixels = case["width"] * case["height"]
    cells = case["size"] / (case["voxel"] * case["ell"])
    blocks, vox = 0.4 * cells * cells, case["ell"] ** 3
    # depth in, keys once, the view out; per block key and indices, and both value rows read, written and given back
    return {"bytes": pixels * (4 + 12 + 4) + blocks * (12 + 16 + vox * 4 * 6), "flops": blocks * vox * 30.0}


# ------------------------------------------------------------------- exact
def exact(case, seed):
    """A fused frame's value rows in float64. Which voxel sees which pixel is decided in float32, step by step, as the
    pipeline defines it; the ray cast depth is a choice among samples and has no such value."""
    if case["kind"] != "frame":
        return None
    frames = _frames(case, seed)
    voxel, ell = case["voxel"], case["ell"]
    limit = _ray(case)[3]
    sets = [_frame_blocks(case, depth, pose, voxel * ell, limit) for depth, pose in frames]
    blocks = sets[-1]
    grid = torch.stack(torch.meshgrid(*[torch.arange(ell, device="cuda")] * 3, indexing="ij"), -1).flip(-1).reshape(-1, 3)
    x = (blocks.long()[:, None, :] * ell + grid).float() * torch.tensor(voxel, dtype=torch.float32, device="cuda")
    d = torch.zeros(x.shape[:2], dtype=torch.float64, device="cuda")
    w = torch.zeros_like(d)
    for (depth, pose), here in zip(frames, sets):
        both = torch.cat([here, blocks])
        _, inverse = torch.unique(both, dim=0, return_inverse=True)
        listed_ = torch.isin(inverse[here.shape[0]:], inverse[:here.shape[0]])
        _integrate_exact(case, x, d, w, listed_, depth, pose, 4 * voxel, limit)
    rows = _frame_rows(case)
    out = torch.zeros((2, rows, ell, ell, ell), dtype=torch.float64, device="cuda")
    u = min(rows, blocks.shape[0])
    out[0, :u] = d[:u].reshape(u, ell, ell, ell)
    out[1, :u] = w[:u].reshape(u, ell, ell, ell)
    return {"blocks": None, "tsdf": out[0], "weight": out[1], "seen": None}


def _f32(v):
    return torch.tensor(v, dtype=torch.float32, device="cuda")


def _frame_blocks(case, depth, pose, edge, limit):
    """int32 [u, 3] distinct block keys of a frame's pixels, in the order in which the pixels meet them."""
    fx, fy, cx, cy = (_f32(v) for v in _camera(case))
    e = pose.cuda()
    row = lambda a, x, y, z: (e[0, a] * x + e[1, a] * y) + e[2, a] * z  # noqa: E731  (R^T v)_a
    v, u = torch.meshgrid(torch.arange(case["height"], device="cuda").float(),
                          torch.arange(case["width"], device="cuda").float(), indexing="ij")
    ok = (depth > 0) & (depth <= _f32(limit))
    z = depth[ok]
    xc, yc = ((u - cx) / fx)[ok] * z, ((v - cy) / fy)[ok] * z
    key = torch.stack([torch.floor((row(a, xc, yc, z) - row(a, e[0, 3], e[1, 3], e[2, 3])) / _f32(edge))
                       for a in range(3)], 1).int()
    distinct, inverse = torch.unique(key, dim=0, return_inverse=True)
    first = torch.full((distinct.shape[0],), key.shape[0], device="cuda", dtype=torch.int64)
    first.scatter_reduce_(0, inverse, torch.arange(key.shape[0], device="cuda"), "amin")
    return distinct[torch.argsort(first)]


def _integrate_exact(case, x, d, w, listed_, depth, pose, trunc, limit):
    fx, fy, cx, cy = (_f32(v) for v in _camera(case))
    e = pose.cuda()
    row = lambda a: ((e[a, 0] * x[..., 0] + e[a, 1] * x[..., 1]) + e[a, 2] * x[..., 2]) + e[a, 3]  # noqa: E731
    xc, yc, zc = row(0), row(1), row(2)
    u = torch.floor(fx * (xc / zc) + cx + 0.5)
    v = torch.floor(fy * (yc / zc) + cy + 0.5)
    ok = listed_[:, None] & (zc > 0) & (u >= 0) & (u < case["width"]) & (v >= 0) & (v < case["height"])
    at = torch.where(ok, v.nan_to_num().clamp(0, case["height"] - 1).long() * case["width"]
                     + u.nan_to_num().clamp(0, case["width"] - 1).long(), 0)
    dm = depth.reshape(-1)[at]
    sdf = dm - zc
    ok &= (dm > 0) & (dm <= _f32(limit)) & (sdf >= -_f32(trunc))
    psi = torch.minimum(sdf, _f32(trunc)).double()
    d.copy_(torch.where(ok, (w * d + psi) / (w + 1), d))
    w.add_(ok.double())
