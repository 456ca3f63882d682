#!/usr/bin/env python
"""Benchmark of the GB300 spatial hash map (ASH hot path) on point-cloud voxelization.

One step = one pass of the hot path over one batch: 4M float32 points of a
synthetic scene are quantised to 5 mm voxel keys, a map of capacity N is
created, the keys are inserted with their point index as value, every point
finds its voxel's buffer index, the live entries are listed and the unique
voxel keys gathered, and the map is destroyed (Sec. 6.1 of the paper).
Metric value = hash ops (insert + find keys) per second over the timed steps.

`--impl reference` times the CPU oracle on a bounded sample of the same
workload instead (the reference arm of this comparison).
"""
import argparse
import ctypes
import datetime
import hashlib
import json
import os
import re
import statistics
import subprocess
import sys
import tempfile
import threading
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

METRIC = "hash ops/s (insert, find) & achieved HBM GB/s vs roofline; p50/p99 served latency"
UNIT = "hash ops/s"
L2_FLUSH_BYTES = 256 << 20
TRACE_EVERY = 4
WORKLOAD = ("point-cloud voxelization: 4M float32 points on 32 spheres + 3 planes in a 10 m cube "
            "(sigma 2 mm), 5 mm voxels, int32x3 keys, capacity = N")


def parse_args(argv=None):
    p = argparse.ArgumentParser()
    p.add_argument("--gpus", type=int, default=1)
    p.add_argument("--steps", type=int, default=1000)
    p.add_argument("--warmup", type=int, default=5)
    p.add_argument("--impl", choices=["ours", "reference"], default="ours")
    p.add_argument("--points", type=int, default=4_000_000)
    p.add_argument("--voxel", type=float, default=0.005)
    p.add_argument("--no-ops", action="store_true", help="skip the per-op figures at the 10^7-key point")
    p.add_argument("--no-cpu", action="store_true", help="skip the cpu_baseline leg")
    p.add_argument("--ops-n", type=int, default=10_000_000)
    p.add_argument("--lean", action="store_true", help="timed steps only (no probe, e2e, per-op or cpu legs)")
    p.add_argument("--no-batched", action="store_true", help="skip the many-map batched comparison")
    p.add_argument("--batched-maps", type=int, default=64)
    p.add_argument("--no-serving", action="store_true", help="skip the serving latency figures")
    p.add_argument("--serving-rates", type=str, default="2000,5000,10000,20000,50000")
    p.add_argument("--serving-requests", type=int, default=10000)
    p.add_argument("--serving-repeats", type=int, default=3)
    p.add_argument("--no-tsdf", action="store_true", help="skip the voxel-block (TSDF) pipeline figures")
    p.add_argument("--no-blocks", action="store_true", help="skip the TSDF-shaped block-map figures")
    p.add_argument("--no-sweep", action="store_true", help="skip the uniqueness sweep")
    p.add_argument("--no-voxel-sizes", action="store_true", help="skip the 5/10/20/50 mm voxel-size sweep")
    p.add_argument("--sweep-only", action="store_true",
                   help="run only the uniqueness sweep (for profiling one of its points) and print its result")
    p.add_argument("--sweep-points", type=str, default="",
                   help="override the sweep points, e.g. 20000000:0.5,1000000:1.0")
    p.add_argument("--block-frames", type=int, default=200)
    p.add_argument("--tsdf-frames", type=int, default=40)
    p.add_argument("--detail", type=str, default=os.path.join(ROOT, "bench_detail.json"),
                   help="file for the full results (sweep, per-op, batched, serving, TSDF, per-kernel figures); "
                        "stdout gets one compact summary line")
    return p.parse_args(argv)


# ----------------------------------------------------------- distribution
def dist_env():
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return world, rank, local


def max_over_ranks(x, world):
    """Max of a float over ranks (identity at world size 1)."""
    if world <= 1:
        return float(x)
    import torch
    import torch.distributed as dist
    dev = "cuda" if dist.get_backend() == "nccl" else "cpu"
    t = torch.tensor([float(x)], dtype=torch.float64, device=dev)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def sum_over_ranks(x, world):
    if world <= 1:
        return float(x)
    import torch
    import torch.distributed as dist
    dev = "cuda" if dist.get_backend() == "nccl" else "cpu"
    t = torch.tensor([float(x)], dtype=torch.float64, device=dev)
    dist.all_reduce(t, op=dist.ReduceOp.SUM)
    return float(t.item())


def aggregate(units_local, seconds_local, world):
    """Whole-job throughput: units summed over ranks / the slowest rank's time."""
    units = sum_over_ranks(units_local, world)
    secs = max_over_ranks(seconds_local, world)
    return units / secs if secs > 0 else 0.0, secs


def barrier(world):
    if world > 1:
        import torch.distributed as dist
        dist.barrier()


# ------------------------------------------------------------------- clocks
class ClockSampler:
    """Samples SM clock and throttle reasons with nvidia-smi while running."""

    FIELDS = ("timestamp,index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index):
        self.gpu = gpu_index
        self.proc = None
        self.path = None
        self.window = None  # (start, end) wall-clock seconds of the timed region

    def mark(self, start, end):
        self.window = (start, end)

    def __enter__(self):
        try:
            fd, self.path = tempfile.mkstemp(suffix=".csv")
            os.close(fd)
            self.proc = subprocess.Popen(
                ["nvidia-smi", "-i", str(self.gpu), f"--query-gpu={self.FIELDS}", "--format=csv,noheader,nounits",
                 "-lms", "50"], stdout=open(self.path, "w"), stderr=subprocess.DEVNULL)
        except Exception:
            self.proc = None
        return self

    def __exit__(self, *exc):
        if self.proc is not None:
            self.proc.terminate()
            try:
                self.proc.wait(timeout=5)
            except Exception:
                self.proc.kill()

    def summary(self):
        if self.proc is None or not self.path or not os.path.exists(self.path):
            return None
        rows = []
        for ln in open(self.path):
            parts = [x.strip() for x in ln.split(",")]
            if len(parts) < 10:
                continue
            try:
                ts = datetime.datetime.strptime(parts[0], "%Y/%m/%d %H:%M:%S.%f").timestamp()
                rows.append((float(parts[2]), float(parts[3]), parts[5:10], ts))
            except ValueError:
                continue
        os.unlink(self.path)
        if self.window is not None:
            inside = [r for r in rows if self.window[0] - 0.06 <= r[3] <= self.window[1] + 0.06]
            in_window = bool(inside)
            rows = inside or rows
        else:
            in_window = False
        if not rows:
            return None
        sm = [r[0] for r in rows]
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        reasons = sorted({names[i] for r in rows for i, v in enumerate(r[2][1:]) if v.lower() == "active"})
        return {"sm_mhz": statistics.median(sm), "sm_max_mhz": max(r[1] for r in rows), "reasons": reasons,
                "samples": len(rows), "samples_in_timed_region": in_window, "interval_ms": 50}


# ------------------------------------------------------ algorithmic bytes
def key_stride(d):
    return 1 if d <= 1 else (2 if d <= 2 else (4 if d <= 4 else 8))


def bytes_find(n_hit, n_miss, d=3):
    """Per key: key row in (4d) + index and mask out (5) + one bucket sector
    (32) + one kB verify sector (32) on a hit."""
    return n_hit * (4 * d + 5 + 64) + n_miss * (4 * d + 5 + 32)


def bytes_claim(n, d=3):
    """Per key: key row in (4d) + one slot sector read and written back (64;
    the bucket load and CAS of the bucket-first claim, the CAS of the
    preferred-slot claim) + slot index out (4)."""
    return n * (4 * d + 68)


def bytes_commit(n, n_win, value_bytes, d=3, heap_identity=True):
    """Per key: slot index in (4) + index and mask out (5) + its winner-flag
    bit (1/8); winners read their key row (4d), write a kB row (4*stride),
    rewrite the slot sector (32) and copy their value rows (read + write),
    and read the heap (4) unless its free part is the identity (a map with
    no erase since create, clear or a compacting rehash)."""
    per_win = 4 * d + 4 * key_stride(d) + 32 + 2 * value_bytes + (0 if heap_identity else 4)
    return n * 9 + (n + 7) // 8 + n_win * per_win


def bytes_list(capacity, n_live, heap_identity=True):
    """A map with no erase since create, clear or a compacting rehash has the
    identity as its heap's free part, so its live indices are 0..t-1 and the
    listing only writes them (4 each).  Otherwise: heap tail read (4 per free
    index), free bitmap cleared, marked and read (c/8 bytes each), live
    indices written (4 each)."""
    if heap_identity:
        return 4 * n_live
    return 4 * (capacity - n_live) + 3 * ((capacity + 7) // 8) + 4 * n_live


def bytes_quantize(n_coords):
    return n_coords * 8


def bytes_gather_keys(n, d=3):
    """Index in (4), kB row read (4*stride; the listing is made of ascending
    runs, so rows are read nearly sequentially), key out (4d)."""
    return n * (4 + 4 * key_stride(d) + 4 * d)


def bytes_erase(n_present, n_absent, d=3):
    """find + the slot rewrite (32) + the heap write (4) for each erased key."""
    return bytes_find(n_present, n_absent, d) + n_present * 36


def split_find(n_hit, n_miss, d=3):
    """bytes_find split into (random, streamed): the bucket sector and, on a
    hit, the kB verify sector are random; the key row in and the index and
    mask out are streamed."""
    n = n_hit + n_miss
    return 32 * n + 32 * n_hit, (4 * d + 5) * n


def split_activate(n, n_win, d=3, heap_identity=True):
    """bytes_claim + bytes_commit (no values) split into (random, streamed):
    the claim's slot sector read and written back (64) and the commit's slot
    rewrite (32 per winner) are random; key rows, slot indices, outputs,
    winner bits, kB rows (written at consecutive indices i = t + rank) and
    heap reads are streamed."""
    total = bytes_claim(n, d) + bytes_commit(n, n_win, 0, d, heap_identity)
    random = 64 * n + 32 * n_win
    return random, total - random


def random_access_fraction(ms, random_bytes, streamed_bytes, random_gbs, copy_gbs):
    """Fraction of the random-access roofline: the time the probe needs for
    the random sectors at the same footprint plus the time a copy needs for
    the streamed bytes, over the measured time.  1.0 means the kernel moves
    its random sectors as fast as the probe and its streamed bytes at copy
    speed."""
    if not random_gbs or not copy_gbs or ms <= 0:
        return None
    bound_s = random_bytes / (random_gbs * 1e9) + streamed_bytes / (copy_gbs * 1e9)
    return bound_s / (ms / 1000.0)


# The sources the insert claim / insert commit / find kernels compile from.
KERNEL_SOURCES = ("ash_device.cuh", "ash_kernels.cuh", "ash_dim.cu")


def _code_only(text):
    """Source text without comments and whitespace runs: a comment edit
    does not change the compiled kernels, so it keeps the digest."""
    text = re.sub(r"/\*.*?\*/", " ", text, flags=re.S)
    text = re.sub(r"//[^\n]*", " ", text)
    return " ".join(text.split())


def source_digest():
    h = hashlib.sha256()
    csrc = os.path.join(ROOT, "paper_2110_00511_gb300", "csrc")
    for f in KERNEL_SOURCES:
        with open(os.path.join(csrc, f), encoding="utf-8") as fh:
            h.update(f.encode())
            h.update(_code_only(fh.read()).encode())
    return h.hexdigest()[:16]


def measured_traffic(kernel):
    """dram bytes per launch from the committed ncu summary, or None if the
    kernel sources changed since it was captured."""
    path = os.path.join(ROOT, "profiles", "traffic.json")
    if not os.path.exists(path):
        return None
    try:
        data = json.load(open(path))
    except Exception:
        return None
    if data.get("source_digest") != source_digest():
        return None
    k = data.get("kernels", {}).get(kernel)
    return None if k is None else k.get("dram_bytes_per_launch_full_size")


def peaks():
    path = os.path.join(ROOT, "MEASURED_PEAKS.json")
    try:
        d = json.load(open(path))
        return float(d["hbm_gbs"]), "measured"
    except Exception:
        return 6800.0, "fallback"


# ------------------------------------------------------------- reference arm
def run_reference(args, world, rank):
    """The reference arm: the CPU oracle, as it stands, over the whole
    voxelization workload on every host core (keys sharded by hash, one
    sequential oracle map per thread; see oracle_all_cores_step)."""
    if rank != 0:
        return 0
    from concurrent.futures import ThreadPoolExecutor
    from paper_2110_00511_gb300 import workloads
    cores = os.cpu_count() or 1
    pts = np.ascontiguousarray(workloads.voxel_scene_points(n=args.points, seed=0))
    with ThreadPoolExecutor(max_workers=cores) as pool:
        for _ in range(args.warmup):
            oracle_all_cores_step(pts, args.voxel, pool, cores)
        t0 = time.perf_counter()
        ops = 0
        for _ in range(args.steps):
            ops += oracle_all_cores_step(pts, args.voxel, pool, cores)
        secs = time.perf_counter() - t0
    value = ops / secs
    sample = f"all {args.points} points per step, keys sharded over {cores} threads (one oracle map each)"
    line = {"impl": "reference", "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": args.gpus,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": 1000 * secs / args.steps,
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "int32",
            "data": "synthetic", "config": {"workload": WORKLOAD, "points": args.points, "voxel_m": args.voxel},
            "cpu_baseline": {"value": value, "unit": UNIT, "cores": cores, "kind": "oracle", "sample": sample},
            "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    emit(line, None)
    return 0


def cpu_baseline(args, pts_np):
    import oracle
    sample_n = min(len(pts_np), 1_000_000)
    pts = pts_np[:sample_n]
    vals = np.arange(sample_n, dtype=np.int32)
    ops = 0
    t0 = time.perf_counter()
    reps = 0
    while True:
        keys = oracle.quantize(pts, args.voxel)
        om = oracle.OracleMap(3, sample_n, [4])
        om.insert(keys, [vals])
        om.find(keys)
        act = om.active_indices()
        _ = om.key_buffer()[act]
        ops += 2 * sample_n
        reps += 1
        el = time.perf_counter() - t0
        if el >= 10.0 or reps >= 40:
            break
    return {"value": ops / el, "unit": UNIT, "cores": 1, "kind": "oracle",
            "sample": f"first {sample_n} points x {reps} passes, 1 thread, {el:.0f} s"}


def _owner(keys, parts):
    """Shard of each int32x3 key: a multiply-xor spatial hash mod parts (the
    partition of keys to host threads; any function of the key works)."""
    k = keys.astype(np.uint32)
    h = (k[:, 0] * np.uint32(73856093)) ^ (k[:, 1] * np.uint32(19349663)) ^ (k[:, 2] * np.uint32(83492791))
    return (h % np.uint32(parts)).astype(np.int64)


def oracle_all_cores_step(pts, voxel, pool, parts):
    """One pass of the voxelization step on `parts` host threads: each thread
    quantises a contiguous slice of the points and hashes its keys to owners;
    then each thread runs its own sequential oracle map over the keys it owns
    (insert with the point index as value, find, listing, key gather).  The
    oracle's C calls release the interpreter lock, so the maps run in
    parallel.  Returns the hash ops done (insert + find keys)."""
    import oracle
    oracle.quantize(pts[:1], voxel)  # loads (and if needed builds) the library before the threads use it
    n = len(pts)
    bounds = np.linspace(0, n, parts + 1).astype(np.int64)

    def front(t):
        lo, hi = bounds[t], bounds[t + 1]
        k = oracle.quantize(pts[lo:hi], voxel)
        own = _owner(k, parts)
        order = np.argsort(own, kind="stable")
        cuts = np.searchsorted(own[order], np.arange(parts + 1))
        ids = np.arange(lo, hi, dtype=np.int32)[order]
        ks = k[order]
        return [(ks[cuts[j]:cuts[j + 1]], ids[cuts[j]:cuts[j + 1]]) for j in range(parts)]

    pieces = list(pool.map(front, range(parts)))

    def back(j):
        kj = np.concatenate([pieces[t][j][0] for t in range(parts)])
        vj = np.concatenate([pieces[t][j][1] for t in range(parts)])
        om = oracle.OracleMap(3, max(1, len(kj)), [4])
        om.insert(kj, [vj])
        om.find(kj)
        act = om.active_indices()
        _ = om.key_buffer()[act]
        return len(kj)

    done = sum(pool.map(back, range(parts)))
    assert done == n
    return 2 * n


def cpu_baseline_all_cores(args, pts_np, budget_s=10.0):
    """The oracle sharded by key over every host core (one sequential map per
    thread), on the same bounded sample as the single-threaded figure."""
    from concurrent.futures import ThreadPoolExecutor
    cores = os.cpu_count() or 1
    sample_n = min(len(pts_np), 1_000_000)
    pts = np.ascontiguousarray(pts_np[:sample_n])
    with ThreadPoolExecutor(max_workers=cores) as pool:
        oracle_all_cores_step(pts, args.voxel, pool, cores)  # warm-up (library load, pools)
        ops, reps = 0, 0
        t0 = time.perf_counter()
        while True:
            ops += oracle_all_cores_step(pts, args.voxel, pool, cores)
            reps += 1
            el = time.perf_counter() - t0
            if el >= budget_s or reps >= 100:
                break
    return {"value": ops / el, "unit": UNIT, "cores": cores, "kind": "oracle",
            "sample": f"first {sample_n} points x {reps} passes, keys sharded over {cores} threads, {el:.0f} s"}


def cpu_baseline_tsdf_frame(c):
    """The CPU oracle on one frame of the voxel-block pipeline (the bench's
    `tsdf` block): block keys, double hash map and integration in full, ray
    casting on every 97th pixel scaled to the image, single-threaded."""
    import oracle
    cam = c["cam"]
    t0 = time.perf_counter()
    okeys = oracle.depth_to_block_keys(c["depth"], c["intr"], c["pose"], c["voxel"] * c["ell"], c["depth_max"])
    olocal = oracle.OracleMap(3, 1 << 17, [4])
    ovol = oracle.OracleMap(3, 1 << 17, [8 * c["ell"] ** 3, 8 * c["ell"] ** 3])
    _, _, ogi = oracle.double_map_activate(olocal, ovol, okeys)
    oracle.tsdf_integrate(ovol, ogi, c["depth"], c["intr"], c["pose"], c["voxel"], c["trunc"], c["depth_max"],
                          ell=c["ell"])
    t_int = time.perf_counter() - t0
    pix = np.arange(0, cam.width * cam.height, 97, dtype=np.int64)
    t0 = time.perf_counter()
    oracle.tsdf_raycast(ovol, c["intr"], c["pose"], cam.width, cam.height, c["voxel"], c["depth_min"], c["step"],
                        c["n_steps"], pixels=pix, ell=c["ell"], value_bytes=8)
    t_rc = (time.perf_counter() - t0) * (cam.width * cam.height) / len(pix)
    return {"ms_per_frame": 1000.0 * (t_int + t_rc), "cores": 1, "kind": "oracle",
            "sample": "frame 0 of the voxel-block pipeline: keys, double map and integration in full; ray casting "
                      "on every 97th pixel, scaled to the image"}


# ------------------------------------------------------------ output line
COMPACT_LIMIT = 1600  # bytes of the one stdout line (well under the 2 KB a log tail keeps)


def _sig(x, digits=4):
    """Floats to `digits` significant digits (keeps the summary line short)."""
    if isinstance(x, float):
        return float(f"{x:.{digits}g}")
    if isinstance(x, dict):
        return {k: _sig(v, digits) for k, v in x.items()}
    if isinstance(x, (list, tuple)):
        return [_sig(v, digits) for v in x]
    return x


def _pick(d, keys):
    if not isinstance(d, dict):
        return None
    return {k: d[k] for k in keys if k in d}


def highlights(full):
    """A few figures of the side blocks for the summary line (G = 10^9):
      graph_G:   the step replayed as a CUDA graph (G hash ops/s);
      sweep:     the largest sweep point beyond 4x L2, activate and find as
                 [G keys/s, fraction of the copy peak, fraction of the
                 random-access roofline, G keys/s in input order]: at a
                 ranged point (keys in home-bucket range order) the
                 roofline fraction is that of the input-order calls;
      batched_G: [batched G ops/s, plain per-map G ops/s, batched p99 ms, plain p99 ms];
      served:  per offered rate [req/s, p99 ms, sequential req/s, sequential p99 ms]."""
    h = {}
    g = full.get("graph_step")
    if isinstance(g, dict) and "value" in g:
        h["graph_G"] = g["value"] / 1e9
    sw = full.get("sweep")
    if isinstance(sw, dict):
        big = [p_ for p_ in sw.get("points", []) if p_.get("working_set_x_l2", 0) >= 4]
        if big:
            p_ = max(big, key=lambda r: r["n"])
            h["sweep"] = {"n": p_["n"], "rho": p_["rho"]}
            for op, short in (("activate", "act"), ("find", "find")):
                r = p_.get(op, {})
                io = r.get("input_order") or r
                h["sweep"][short] = [(r.get("keys_per_s") or 0) / 1e9, r.get("frac_hbm"),
                                     io.get("frac_random_access_roofline"), (io.get("keys_per_s") or 0) / 1e9]
    b = full.get("batched")
    if isinstance(b, dict) and "batched_graph" in b:
        h["batched_G"] = [b["batched_graph"]["ops_per_s"] / 1e9, b["plain_per_map"]["ops_per_s"] / 1e9,
                        b["batched_graph"]["ms_p99"], b["plain_per_map"]["ms_p99"]]
    sv = full.get("serving")
    if isinstance(sv, dict) and isinstance(sv.get("rates"), dict):
        mode = sv.get("default_mode", "served")
        rows = {"mode": mode}
        for rate, e in sv["rates"].items():
            s_, q_ = e.get(mode) or {}, e.get("sequential_plain") or {}
            rows[rate] = [s_.get("req_per_s"), s_.get("p99_ms"), q_.get("req_per_s"), q_.get("p99_ms")]
        h["served"] = rows
    return h


def compact_line(full, detail_path=None):
    """The one stdout line: the contract's keys, the roofline, the CPU
    baseline, the end-to-end figure, clocks and a few highlights.  Everything
    else goes to the detail file."""
    out = _pick(full, ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better",
                       "scaling", "vs_baseline", "dtype", "data", "gpu_launches"))
    if "impl" in full:
        out = {"impl": full["impl"], **out}
    out["config"] = _pick(full.get("config") or {}, ("workload", "points", "voxel_m", "unique_voxels", "l2",
                                                     "parallelism", "sample"))
    rl = full.get("roofline")
    out["roofline"] = _pick(rl, ("bound", "kernel", "achieved", "peak", "unit", "frac", "traffic")) if rl else None
    if isinstance(rl, dict) and rl.get("peak_kind"):
        out["roofline"]["peak_kind"] = rl["peak_kind"].split(" ")[0]
    cpu = full.get("cpu_baseline")
    if isinstance(cpu, dict):
        out["cpu_baseline"] = _pick(cpu, ("value", "unit", "cores", "kind", "sample"))
        if isinstance(cpu.get("all_cores"), dict):
            out["cpu_baseline"]["all_cores"] = _pick(cpu["all_cores"], ("value", "cores"))
    else:
        out["cpu_baseline"] = None
    e2e = full.get("e2e")
    out["e2e"] = _pick(e2e, ("value", "unit", "h2d_bytes_per_step", "d2h_bytes_per_step", "error")) \
        if isinstance(e2e, dict) else None
    clk = full.get("clocks")
    out["clocks"] = _pick(clk, ("sm_mhz", "sm_max_mhz", "reasons", "samples_in_timed_region")) \
        if isinstance(clk, dict) else None
    hl = highlights(full)
    if hl:
        out["highlights"] = hl
    if detail_path:
        out["detail"] = os.path.basename(detail_path)
    out = _sig(out)
    line = json.dumps(out, separators=(",", ":"))
    for drop in ("served_rows", "batched_G", "all"):
        if len(line) <= COMPACT_LIMIT or "highlights" not in out:
            break
        h = out["highlights"]
        if drop == "served_rows" and "served" in h:
            rates = [k for k in h["served"] if k != "mode"]
            h["served"] = {k: h["served"][k] for k in ["mode"] + rates[:1] + rates[-1:]}
        elif drop == "all":
            out.pop("highlights")
        else:
            h.pop(drop, None)
        line = json.dumps(out, separators=(",", ":"))
    if len(line) > COMPACT_LIMIT:
        for k in ("config", "cpu_baseline"):
            if isinstance(out.get(k), dict):
                for kk in ("workload", "sample"):
                    if isinstance(out[k].get(kk), str):
                        out[k][kk] = out[k][kk][:120]
        line = json.dumps(out, separators=(",", ":"))
    return line


def emit(full, detail_path):
    """Writes the full results to detail_path (if given) and prints the
    compact summary line last on stdout."""
    if detail_path:
        try:
            with open(detail_path, "w") as fh:
                json.dump(full, fh, indent=1)
        except OSError as e:
            print(f"bench: could not write {detail_path}: {e}", file=sys.stderr)
            detail_path = None
    print(compact_line(full, detail_path), flush=True)


# ------------------------------------------------------------------ GPU arm
def main(argv=None):
    args = parse_args(argv)
    world, rank, local = dist_env()
    if args.impl == "reference":
        return run_reference(args, world, rank)

    import torch
    from paper_2110_00511_gb300 import ash, build, workloads

    if world > 1:
        import torch.distributed as dist
        torch.cuda.set_device(local)
        dist.init_process_group("nccl", device_id=torch.device("cuda", local))
    else:
        torch.cuda.set_device(0)
    device = torch.device("cuda", torch.cuda.current_device())
    if rank == 0 or not build.up_to_date():
        build.build()
    barrier(world)
    ash.lib()
    if args.sweep_only:
        hbm_peak, _ = peaks()
        res = sweep_figures(args, device, hbm_peak)
        if rank == 0:
            print(json.dumps(_sig(res)), flush=True)
        return 0

    N = args.points
    pts_np = workloads.voxel_scene_points(n=N, seed=rank)
    pts = torch.from_numpy(pts_np).to(device)
    point_ids = torch.arange(N, dtype=torch.int32, device=device)
    keys = torch.empty((N, 3), dtype=torch.int32, device=device)
    flush = torch.empty(L2_FLUSH_BYTES, dtype=torch.uint8, device=device)
    stream = torch.cuda.current_stream()

    aux = torch.cuda.Stream(device=device)

    def step(points, keys_out, voxel=args.voxel):
        # No host synchronisation anywhere in the step: the live count stays on
        # the device and bounds the gather of the unique voxel keys.  Two
        # streams overlap independent work: the map is created (table fill,
        # heap init) while the points are quantised, and the live entries are
        # listed and gathered while every point finds its voxel.
        main = torch.cuda.current_stream(device)
        aux.wait_stream(main)
        with torch.cuda.stream(aux):
            hm = ash.HashMap(3, N, [(1,)], [torch.int32], device=device)
        ash.ash_quantize(points, voxel, out=keys_out)
        main.wait_stream(aux)
        idx, mask = hm.insert(keys_out, [point_ids])
        aux.wait_stream(main)
        with torch.cuda.stream(aux):
            act, count = hm.active_indices_async()
            uniq = hm.gather_keys_count(act, count)
        fidx, fmask = hm.find(keys_out)  # last call on the main stream
        main.wait_stream(aux)            # join before the map is freed on the main stream
        del hm
        return fidx, uniq, count

    def step_fused(points):
        # The same step with the quantisation done inside the hash kernels
        # (insert / find on the float32 points): no key array is written.
        main = torch.cuda.current_stream(device)
        aux.wait_stream(main)
        with torch.cuda.stream(aux):
            hm = ash.HashMap(3, N, [(1,)], [torch.int32], device=device)
        main.wait_stream(aux)
        hm.insert_points(points, args.voxel, [point_ids])
        aux.wait_stream(main)
        with torch.cuda.stream(aux):
            act, count = hm.active_indices_async()
            uniq = hm.gather_keys_count(act, count)
        fidx, fmask = hm.find_points(points, args.voxel)
        main.wait_stream(aux)
        del hm
        return fidx, uniq, count

    def step_zero_copy(host_pts, host_idx, host_mask, host_uniq, host_cnt):
        # The same step reading the points from host memory and writing the
        # per-point indices and masks, the unique voxel keys and their count to
        # host memory, directly from the kernels (a coherent CPU-GPU system:
        # pageable memory access), with no staging copies.
        lib = ash.lib()
        main = torch.cuda.current_stream(device)
        ms = ctypes.c_void_p(main.cuda_stream)
        aux.wait_stream(main)
        with torch.cuda.stream(aux):
            hm = ash.HashMap(3, N, [(1,)], [torch.int32], device=device)
        ash._check(lib.ash_quantize(ash._ptr(host_pts), host_pts.numel(), ctypes.c_float(args.voxel),
                                    ash._ptr(keys), ms))
        main.wait_stream(aux)
        hm.insert(keys, [point_ids])
        aux.wait_stream(main)
        with torch.cuda.stream(aux):
            act, count = hm.active_indices_async()
            ash._check(lib.ash_gather_keys_count(hm.handle, ash._ptr(act), N, ash._ptr(count), ash._ptr(host_uniq),
                                                 ctypes.c_void_p(aux.cuda_stream)))
            host_cnt.copy_(count, non_blocking=True)
        ash._check(lib.ash_find(hm.handle, ash._ptr(keys), N, ash._ptr(host_idx), ash._ptr(host_mask), ms))
        main.wait_stream(aux)
        del hm

    import gc
    clocks = ClockSampler(local)
    clocks.__enter__()  # started before warm-up so its start-up is outside the timed steps
    for _ in range(args.warmup):
        step(pts, keys)
    torch.cuda.synchronize()

    # ------------------------------------------------------------ timed steps
    ash.ash_trace_reset()
    starts = [torch.cuda.Event(enable_timing=True) for _ in range(args.steps)]
    ends = [torch.cuda.Event(enable_timing=True) for _ in range(args.steps)]
    n_unique = 0
    barrier(world)
    torch.cuda.synchronize()
    launches0 = ash.ash_kernel_launch_count()
    t_wall0 = time.time()
    gc.disable()
    for s in range(args.steps):
        flush.zero_()
        # per-kernel events on every TRACE_EVERY-th timed step: the kernel
        # durations come from the timed region without adding an event pair
        # to every launch of every step
        ash.ash_trace_enable(s % TRACE_EVERY == 0)
        starts[s].record(stream)
        _, uniq, count = step(pts, keys)
        ends[s].record(stream)
    ash.ash_trace_enable(False)
    torch.cuda.synchronize()
    t_wall1 = time.time()
    n_unique = int(count.item())
    gc.enable()
    clocks.mark(t_wall0, t_wall1)
    clocks.__exit__(None, None, None)
    barrier(world)
    launches = ash.ash_kernel_launch_count() - launches0
    step_ms = [a.elapsed_time(b) for a, b in zip(starts, ends)]
    secs_local = sum(step_ms) / 1000.0
    ops_per_step = 2 * N
    value, secs = aggregate(ops_per_step * args.steps, secs_local, world)
    trace = ash.ash_trace_collect()

    # ---------------------------------------------------------- roofline
    hbm_peak, peak_kind = peaks()
    per_launch_bytes = {
        "quantize": bytes_quantize(3 * N),
        "insert_claim": bytes_claim(N),
        "insert_commit": bytes_commit(N, n_unique, 4),
        "find": bytes_find(N, 0),
        "list_active": bytes_list(N, n_unique),
        "gather_keys": bytes_gather_keys(n_unique),
        "storage_init": (16 + 4 + 4) * N + N // 8 + 32,  # table, heap, values, winner flags, counters
    }
    kernels = {}
    total_kernel_ms = sum(ms for ms, n in trace.values())
    for name, (ms, n) in trace.items():
        if n == 0:
            continue
        k = {"traced_launches": n, "ms_per_launch": ms / n,
             "share": ms / total_kernel_ms if total_kernel_ms else 0.0}
        if name in per_launch_bytes:
            gbs = per_launch_bytes[name] / (ms / n / 1000.0) / 1e9
            k.update({"algo_bytes_per_launch": per_launch_bytes[name], "achieved_gbs": gbs, "frac": gbs / hbm_peak})
        kernels[name] = k
    dominant = max((k for k in kernels if "achieved_gbs" in kernels[k]), key=lambda k: kernels[k]["share"])
    dk = kernels[dominant]
    roofline = {"bound": "hbm", "kernel": dominant, "achieved": dk["achieved_gbs"], "peak": hbm_peak,
                "peak_kind": peak_kind + " (MEASURED_PEAKS.json hbm_gbs, copy bandwidth)" if peak_kind == "measured" else peak_kind,
                "unit": "GB/s", "frac": dk["achieved_gbs"] / hbm_peak,
                "traffic": measured_traffic(dominant)}

    # the two hash operations of the step, each over all of its kernels
    op_roofline = {}
    for op, parts in (("insert", ("insert_claim", "insert_commit")), ("find", ("find",))):
        if all(p_ in kernels and "algo_bytes_per_launch" in kernels[p_] for p_ in parts):
            nbytes = sum(kernels[p_]["algo_bytes_per_launch"] for p_ in parts)
            ms_op = sum(kernels[p_]["ms_per_launch"] for p_ in parts)
            gbs = nbytes / (ms_op / 1000.0) / 1e9
            op_roofline[op] = {"kernels": list(parts), "algo_bytes": nbytes, "ms": ms_op,
                               "keys_per_s": N / (ms_op / 1000.0), "achieved_gbs": gbs, "frac": gbs / hbm_peak}

    # ----------------------------------------------- random-access rooflines
    # Measured by the library's own probe kernels: random sector reads at the
    # step's table footprint (64 MB), at 512 MiB and at 8 GiB; random 64-bit
    # CAS and the claim's load->CAS chain at the table footprint.  The insert
    # claim is bound by the atomic chain, the find by random reads.
    probe = None
    try:
        if args.lean:
            raise RuntimeError("skipped (--lean)")
        sink = torch.zeros(4096, dtype=torch.int32, device=device)
        probe = {}

        def timed_probe(fn, reps=3):
            best = None
            for _ in range(reps):
                e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                e0.record()
                fn()
                e1.record()
                torch.cuda.synchronize()
                ms = e0.elapsed_time(e1)
                best = ms if best is None else min(best, ms)
            return best

        table_bytes = 16 * N  # 2 slots of 8 bytes per unit of capacity
        for label, nbytes in (("table", table_bytes), ("512MiB", 512 << 20), ("8GiB", 8 << 30)):
            buf = torch.empty(nbytes, dtype=torch.uint8, device=device)
            n_reads = 1 << 26
            best = None
            for loads in (4, 8, 16):
                ms = timed_probe(lambda: ash.ash_probe_random_read(buf, n_reads, 32, sink, seed=7,
                                                                   loads_per_thread=loads))
                probe[f"read32_{label}_loads{loads}_Gops"] = n_reads / (ms / 1000) / 1e9
                best = ms if best is None else min(best, ms)
            probe[f"read32_{label}_Gops"] = n_reads / (best / 1000) / 1e9
            probe[f"read32_{label}_GBps"] = n_reads * 32 / (best / 1000) / 1e9
            del buf
        tbl = torch.empty(table_bytes, dtype=torch.uint8, device=device)
        n_ops = N
        for mode, label in ((0, "cas_table_Gops"), (1, "load_cas_chain_table_Gops")):
            # the slots start all ones (EMPTY); the fill stays outside the events
            best = None
            for _ in range(3):
                tbl.fill_(255)
                torch.cuda.synchronize()
                e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                e0.record()
                ash.ash_probe_random_atomic(tbl, n_ops, mode, sink, seed=11)
                e1.record()
                torch.cuda.synchronize()
                ms = e0.elapsed_time(e1)
                best = ms if best is None else min(best, ms)
            probe[label] = n_ops / (best / 1000) / 1e9
        del tbl
        claim_rate = N / (kernels["insert_claim"]["ms_per_launch"] / 1000) / 1e9
        find_sectors = 2 * N / (kernels["find"]["ms_per_launch"] / 1000) / 1e9
        probe["insert_claim_Gkeys"] = claim_rate
        probe["insert_claim_frac_of_load_cas_chain"] = claim_rate / probe["load_cas_chain_table_Gops"]
        probe["find_random_sectors_G"] = find_sectors
        probe["find_frac_of_read32_table"] = find_sectors / probe["read32_table_Gops"]
    except Exception as e:  # noqa: BLE001
        probe = {"error": str(e)[:200]}

    # ---------------------------------------------------------------- e2e
    e2e = None
    try:
        if args.lean:
            raise RuntimeError("skipped (--lean)")
        host_pts = torch.from_numpy(pts_np).pin_memory()
        host_idx = [torch.empty(N, dtype=torch.int32).pin_memory() for _ in range(2)]
        host_uniq = [torch.empty((N, 3), dtype=torch.int32).pin_memory() for _ in range(2)]
        host_cnt = [torch.empty(1, dtype=torch.int64).pin_memory() for _ in range(2)]
        dev_pts = [torch.empty_like(pts) for _ in range(2)]
        s_in = torch.cuda.Stream(device=device)
        s_out = torch.cuda.Stream(device=device)
        e2e_steps = max(4, min(args.steps, 20))

        def pipelined(K):
            # three stages on their own streams, two buffers: the upload of
            # step k+1 and the download of step k-1 overlap step k's kernels;
            # every step's own copies are inside the timed region
            main = torch.cuda.current_stream(device)
            ev_in = [torch.cuda.Event() for _ in range(2)]
            ev_comp = [torch.cuda.Event() for _ in range(2)]
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record(s_in)
            for k in range(K):
                b = k % 2
                if k >= 2:
                    s_in.wait_event(ev_comp[b])        # step k-2 no longer reads dev_pts[b]
                with torch.cuda.stream(s_in):
                    dev_pts[b].copy_(host_pts, non_blocking=True)
                ev_in[b].record(s_in)
                main.wait_event(ev_in[b])
                fidx, uniq, cnt = step(dev_pts[b], keys)
                ev_comp[b].record(main)
                s_out.wait_event(ev_comp[b])
                with torch.cuda.stream(s_out):
                    for t_ in (fidx, uniq, cnt):
                        t_.record_stream(s_out)
                    host_idx[b].copy_(fidx, non_blocking=True)
                    host_uniq[b].copy_(uniq, non_blocking=True)  # N-row bound; the first count rows are valid
                    host_cnt[b].copy_(cnt, non_blocking=True)
            s_out.wait_event(ev_comp[(K - 1) % 2])
            e1.record(s_out)
            torch.cuda.synchronize()
            return e0.elapsed_time(e1)

        flush.zero_()
        pipelined(2)  # warms the pinned path and the streams
        flush.zero_()
        torch.cuda.synchronize()
        ms_total = pipelined(e2e_steps)
        d2h = 4 * N + 12 * N + 8
        e2e_secs = max_over_ranks(ms_total / 1000.0, world)
        e2e = {"value": sum_over_ranks(ops_per_step * e2e_steps, world) / e2e_secs, "unit": UNIT,
               "h2d_bytes_per_step": 12 * N, "d2h_bytes_per_step": d2h,
               "path": "pinned host buffers; per step an upload of the points and a download of the per-point "
                       "indices, unique keys and count, pipelined over two buffers on separate copy streams",
               "steps": e2e_steps}
        # zero-copy variant: the kernels read and write host memory directly
        if ash.ash_get_device_info(device.index)["pageable_memory_access"] == 1:
            zc_idx = torch.empty(N, dtype=torch.int32).pin_memory()
            zc_mask = torch.empty(N, dtype=torch.uint8).pin_memory()
            zc_uniq = torch.empty((N, 3), dtype=torch.int32).pin_memory()
            zc_cnt = torch.empty(1, dtype=torch.int64).pin_memory()
            ms_zc = 0.0
            for s in range(e2e_steps + 1):
                flush.zero_()
                e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                e0.record(stream)
                step_zero_copy(host_pts, zc_idx, zc_mask, zc_uniq, zc_cnt)
                e1.record(stream)
                torch.cuda.synchronize()
                if s > 0:
                    ms_zc += e0.elapsed_time(e1)
            last = (e2e_steps - 1) % 2
            n_u = int(zc_cnt[0])

            def packed_sorted(u, k):
                u = u[:k].to(device).to(torch.int64) + (1 << 20)
                return torch.sort((u[:, 0] << 42) | (u[:, 1] << 21) | u[:, 2]).values
            # buffer indices differ between runs (allocation order); the unique
            # key sets, the count and the masks must not
            ok = (n_u == n_unique == int(host_cnt[last][0]) and bool(zc_mask.bool().all())
                  and bool(torch.equal(packed_sorted(zc_uniq, n_u), packed_sorted(host_uniq[last], n_u))))
            zc_secs = max_over_ranks(ms_zc / 1000.0, world)
            e2e["zero_copy"] = {"value": sum_over_ranks(ops_per_step * e2e_steps, world) / zc_secs, "unit": UNIT,
                                "h2d_bytes_per_step": 12 * N, "d2h_bytes_per_step": 5 * N + 12 * n_u + 8,
                                "path": "kernels read the points from and write the outputs to pinned host "
                                        "memory directly (coherent CPU-GPU memory), no staging copies; steps "
                                        "one after another (not pipelined)",
                                "outputs_equal_staged": ok}
    except Exception as e:  # noqa: BLE001
        e2e = {"error": str(e)[:200]}

    # ------------------------------------- the step replayed as a CUDA graph
    graph_step = None
    try:
        if args.lean:
            raise RuntimeError("skipped (--lean)")
        cap = torch.cuda.Stream(device=device)
        cap.wait_stream(stream)
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=cap):
            _, _, g_count = step(pts, keys)
        torch.cuda.synchronize()
        gms = []
        for s in range(min(args.steps, 200) + 3):
            flush.zero_()
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record(stream)
            g.replay()
            e1.record(stream)
            if s >= 3:
                gms.append((e0, e1))
        torch.cuda.synchronize()
        gt = [a.elapsed_time(b) for a, b in gms]
        graph_step = {"ms_median": statistics.median(gt), "ms_min": min(gt),
                      "value": ops_per_step / (statistics.median(gt) / 1000.0), "unit": UNIT,
                      "replays": len(gt), "unique_voxels": int(g_count.item()),
                      "note": "the same step (map creation, quantize, insert, find, listing, gather, destroy) "
                              "captured once and replayed; memory comes from graph allocation nodes"}
        del g
    except Exception as e:  # noqa: BLE001
        graph_step = {"error": str(e)[:200]}

    # ------------------------------------ the step with in-kernel quantisation
    fused = None
    try:
        if args.lean:
            raise RuntimeError("skipped (--lean)")
        for _ in range(3):
            step_fused(pts)
        torch.cuda.synchronize()
        fev = []
        for s in range(min(args.steps, 300)):
            flush.zero_()
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record(stream)
            _, _, f_count = step_fused(pts)
            e1.record(stream)
            fev.append((e0, e1))
        torch.cuda.synchronize()
        ft = [a.elapsed_time(b) for a, b in fev]
        fused = {"ms_median": statistics.median(ft), "ms_min": min(ft),
                 "value": ops_per_step / (statistics.median(ft) / 1000.0), "unit": UNIT, "steps": len(ft),
                 "unique_voxels": int(f_count.item()),
                 "note": "insert and find take the float32 points and quantise them in the kernels "
                         "(ash_insert_points / ash_find_points); outputs as the headline step"}
    except Exception as e:  # noqa: BLE001
        fused = {"error": str(e)[:200]}

    # ---------------------------- the paper's voxel sizes (Sec. 6.1): 5-50 mm
    voxel_sizes = None
    if not args.lean and not args.no_voxel_sizes:
        try:
            voxel_sizes = voxel_size_figures(step, pts, keys, flush, N, hbm_peak, stream)
        except Exception as e:  # noqa: BLE001
            voxel_sizes = {"error": str(e)[:300]}

    # ------------------------------------------------- per-op figures (10^7)
    ops = None
    if not args.no_ops and not args.lean:
        ops = per_op_figures(args, device, hbm_peak)

    batched = None
    if not args.no_batched and not args.lean:
        batched = batched_figures(args, device)

    serving = None
    if not args.no_serving and not args.lean:
        serving = serving_figures(args, device)

    sweep = None
    if not args.no_sweep and not args.lean:
        try:
            sweep = sweep_figures(args, device, hbm_peak)
        except Exception as e:  # noqa: BLE001
            sweep = {"error": str(e)[:300]}

    blocks = None
    if not args.no_blocks and not args.lean:
        try:
            blocks = tsdf_block_map_figures(args, device, hbm_peak)
        except Exception as e:  # noqa: BLE001
            blocks = {"error": str(e)[:300]}

    tsdf, tsdf_cpu_inputs = None, None
    if not args.no_tsdf and not args.lean:
        try:
            tsdf, tsdf_cpu_inputs = tsdf_figures(args, device, hbm_peak, rank == 0 and world == 1 and not args.no_cpu)
        except Exception as e:  # noqa: BLE001
            tsdf, tsdf_cpu_inputs = {"error": str(e)[:300]}, None

    cpu = None
    if rank == 0 and world == 1 and not args.no_cpu and not args.lean:
        cpu = cpu_baseline(args, pts_np)
        try:
            cpu["all_cores"] = cpu_baseline_all_cores(args, pts_np)
        except Exception as e:  # noqa: BLE001
            cpu["all_cores"] = {"error": str(e)[:200]}
        if tsdf_cpu_inputs is not None:
            cpu["tsdf_frame"] = cpu_baseline_tsdf_frame(tsdf_cpu_inputs)

    if rank == 0:
        full = {"metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": args.steps,
                "warmup": args.warmup, "ms_per_step": 1000.0 * secs / args.steps, "higher_is_better": True,
                "scaling": "weak", "vs_baseline": None, "dtype": "int32", "data": "synthetic",
                "config": {"workload": WORKLOAD, "points": N, "voxel_m": args.voxel, "key_dim": 3,
                           "unique_voxels": n_unique, "value": "int32 point index",
                           "step": "quantize || create, insert, find || (list active, gather unique keys), destroy "
                                   "(two streams, no host synchronisation inside a step)",
                           "l2": "flushed (256 MiB write) between steps",
                           "parallelism": f"replicas x{world}" if world > 1 else "single GPU"},
                "gpu_launches": launches, "roofline": roofline, "cpu_baseline": cpu, "e2e": e2e,
                "graph_step": graph_step, "fused_quantize_step": fused,
                "clocks": clocks.summary(), "kernels": kernels, "hash_op_roofline": op_roofline,
                "random_access_roofline": probe,
                "step_ms": {"median": statistics.median(step_ms), "min": min(step_ms), "max": max(step_ms)},
                "voxel_sizes": voxel_sizes, "ops": ops, "batched": batched, "serving": serving, "sweep": sweep, "tsdf_block_map": blocks, "tsdf": tsdf,
                "source_digest": source_digest()}
        emit(full, args.detail)
    if world > 1:
        import torch.distributed as dist
        dist.destroy_process_group()
    return 0


def voxel_size_figures(step, pts, keys, flush, N, hbm_peak, stream, sizes=(0.005, 0.01, 0.02, 0.05), reps=30):
    """The voxelization step at the paper's voxel sizes (Sec. 6.1: 5, 10, 20
    and 50 mm) on the same 4M points: larger voxels mean more points per
    voxel, so more of the insert's keys are duplicates that join an earlier
    claim and lose.  Per size: unique voxels, median step time, hash ops/s,
    and insert (claim + commit) and find as fractions of the copy peak by
    algorithmic bytes, from per-kernel events."""
    import torch
    from paper_2110_00511_gb300 import ash
    out = {"points": N, "sizes": []}
    for vs in sizes:
        for _ in range(3):
            step(pts, keys, voxel=vs)
        torch.cuda.synchronize()
        ash.ash_trace_reset()
        ev = []
        for r in range(reps):
            ash.ash_trace_enable(r % TRACE_EVERY == 0)  # per-kernel events on every 4th step only
            flush.zero_()
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record(stream)
            _, _, count = step(pts, keys, voxel=vs)
            e1.record(stream)
            ev.append((e0, e1))
        ash.ash_trace_enable(False)
        torch.cuda.synchronize()
        tr = ash.ash_trace_collect()
        n_unique = int(count.item())
        ms = statistics.median(a.elapsed_time(b) for a, b in ev)
        k_ms = {k: t / n for k, (t, n) in tr.items() if n}
        rec = {"voxel_m": vs, "unique_voxels": n_unique, "points_per_voxel": N / max(1, n_unique),
               "step_ms": ms, "hash_ops_per_s": 2 * N / (ms / 1000.0),
               "kernel_ms": {k: k_ms[k] for k in ("quantize", "insert_claim", "insert_commit", "find") if k in k_ms}}
        if "insert_claim" in k_ms and "insert_commit" in k_ms:
            b_ins = bytes_claim(N) + bytes_commit(N, n_unique, 4)
            t_ins = (k_ms["insert_claim"] + k_ms["insert_commit"]) / 1000.0
            rec["insert"] = {"keys_per_s": N / t_ins, "algo_gbs": b_ins / t_ins / 1e9,
                             "frac_hbm": b_ins / t_ins / 1e9 / hbm_peak}
        if "find" in k_ms:
            b_f = bytes_find(N, 0)
            t_f = k_ms["find"] / 1000.0
            rec["find"] = {"keys_per_s": N / t_f, "algo_gbs": b_f / t_f / 1e9, "frac_hbm": b_f / t_f / 1e9 / hbm_peak}
        out["sizes"].append(rec)
    return out


def device_uniform_keys(n, rho, seed, device):
    """n int32x3 keys with round(rho n) distinct values, drawn on the device:
    U distinct keys uniform in [-2^20, 2^20)^3 (collisions in a 2^63 space
    are negligible and the map counts the real number), each appearing once,
    the rest uniform picks among them, shuffled.  The shape of the sweep's
    generator in workloads.uniform_keys, for sizes where host generation
    would dominate the run."""
    import torch
    g = torch.Generator(device=device)
    g.manual_seed(seed)
    u = max(1, int(round(rho * n)))
    distinct = torch.randint(-(1 << 20), 1 << 20, (u, 3), generator=g, device=device, dtype=torch.int32)
    pick = torch.cat([torch.arange(u, device=device),
                      torch.randint(0, u, (n - u,), generator=g, device=device)])
    pick = pick[torch.randperm(n, generator=g, device=device)]
    return distinct[pick].contiguous()


def probe_random_gbs(buf_bytes, device, reps=3):
    """Random 32-byte sector reads over a buffer of buf_bytes, best over 8 and
    16 loads in flight per thread and `reps` runs: (GB/s, G sectors/s)."""
    import torch
    from paper_2110_00511_gb300 import ash
    buf = torch.empty(max(64, (buf_bytes + 63) // 64 * 64), dtype=torch.uint8, device=device)
    sink = torch.zeros(4096, dtype=torch.int32, device=device)
    n_reads = 1 << 26
    best = None
    for loads in (8, 16):
        for _ in range(reps):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record()
            ash.ash_probe_random_read(buf, n_reads, 32, sink, seed=17, loads_per_thread=loads)
            e1.record()
            torch.cuda.synchronize()
            ms = e0.elapsed_time(e1)
            best = ms if best is None else min(best, ms)
    del buf
    return n_reads * 32 / (best / 1000.0) / 1e9, n_reads / (best / 1000.0) / 1e9


def small_call_figures(keys, queries, n, device, flush, calls=64):
    """Per-call cost of small batches (microseconds), L2 flushed before each
    single call:
      python:        CUDA events around one HashMap call (host time of the
                     binding and the library included, as the sweep times it);
      abi:           events around one call of the C ABI with outputs
                     allocated beforehand (the library's host time and its
                     kernels);
      gpu:           the same C ABI call queued behind a GPU sleep, so that
                     the host's work is hidden: the device time of the call;
      pipelined:     `calls` calls issued back to back through HashMap
                     (activate on as many fresh maps, find on one map), total
                     time / calls: the cost per call when the host keeps the
                     stream busy;
      abi_pipelined: the same through the C ABI.
    floor_us: the python and gpu timings of one PyTorch call that launches a
    single tiny kernel (a 16-element fill): what any one-kernel call costs in
    this harness."""
    import torch
    from paper_2110_00511_gb300 import ash
    L = ash.lib()
    idx = torch.empty(n, dtype=torch.int32, device=device)
    msk = torch.empty(n, dtype=torch.bool, device=device)
    st = ash._stream_of(device.index)

    def ev_span(fn, reps=5, hide_host=False):
        best = None
        for _ in range(reps):
            flush.zero_()
            torch.cuda.synchronize()
            if hide_host:
                torch.cuda._sleep(2_000_000)  # about 1 ms: the call is queued before the GPU reaches it
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record()
            fn()
            e1.record()
            torch.cuda.synchronize()
            best = e0.elapsed_time(e1) if best is None else min(best, e0.elapsed_time(e1))
        return 1000.0 * best

    def back_to_back(fns):
        torch.cuda.synchronize()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        for fn in fns:
            fn()
        e1.record()
        torch.cuda.synchronize()
        return 1000.0 * e0.elapsed_time(e1) / len(fns)

    out = {}
    tiny = torch.empty(16, dtype=torch.int32, device=device)
    out["floor_us"] = {"python_one_kernel": ev_span(lambda: tiny.zero_()),
                       "gpu_one_kernel": ev_span(lambda: tiny.zero_(), hide_host=True)}
    fresh = []

    def fresh_map():
        fresh.append(ash.HashMap(3, n, device=device))
        torch.cuda.synchronize()
        return fresh[-1]

    def abi_activate(m):
        return lambda: L.ash_activate(m.handle, keys.data_ptr(), n, idx.data_ptr(), msk.data_ptr(), st)

    res = {}
    for name in ("python", "abi", "gpu"):
        best = None
        for _ in range(5):
            m = fresh_map()
            if name == "python":
                us = ev_span(lambda: m.activate(keys), reps=1)
            else:
                us = ev_span(abi_activate(m), reps=1, hide_host=name == "gpu")
            best = us if best is None else min(best, us)
        res[name] = best
    maps = [ash.HashMap(3, n, device=device) for _ in range(calls)]
    res["pipelined"] = back_to_back([(lambda m=m: m.activate(keys)) for m in maps])
    maps2 = [ash.HashMap(3, n, device=device) for _ in range(calls)]
    res["abi_pipelined"] = back_to_back([abi_activate(m) for m in maps2])
    out["activate_us"] = res
    m = maps[0]
    abi_find = lambda: L.ash_find(m.handle, queries.data_ptr(), n, idx.data_ptr(), msk.data_ptr(), st)
    res = {"python": ev_span(lambda: m.find(queries)), "abi": ev_span(abi_find),
           "gpu": ev_span(abi_find, hide_host=True),
           "pipelined": back_to_back([lambda: m.find(queries)] * calls),
           "abi_pipelined": back_to_back([abi_find] * calls)}
    out["find_us"] = res
    del maps, maps2, fresh
    return out


def sweep_figures(args, device, hbm_peak):
    """The uniqueness sweep of the voxelization setting (Sec. 5.1 / 6.1
    shape): n uniform int32x3 keys at uniqueness rho, capacity n, activate of
    the keys, then find of the same keys in a fresh random order (so the kB
    verify of a hit is a random access, as the byte model counts it), L2
    flushed before each timed call.  Each point reports ops/s, algorithmic
    GB/s, the fraction of the HBM copy peak, and the fraction of the
    random-access roofline: the random-sector read probe run over a buffer of
    the point's own random-access footprint (the buckets and kB rows of its
    distinct keys; a point whose footprint fits in L2 gets none) gives the
    rate for the random sectors, the copy peak the rate for the streamed bytes (see
    random_access_fraction).

    Points whose table is larger than 1.5 times L2 (2^20 keys or more) run, by
    default, with the keys in home-bucket range order (tuning
    partition_keys): their random accesses are then local to one range at a
    time, so the random-access roofline no longer bounds them.  Those points
    also time both calls in input order (partition_keys = 1), report the
    random-access fraction for that variant, and give the ranged calls'
    speed-up over it."""
    import torch
    from paper_2110_00511_gb300 import ash
    l2 = torch.cuda.get_device_properties(device).L2_cache_size
    flush = torch.empty(L2_FLUSH_BYTES, dtype=torch.uint8, device=device)
    if args.sweep_points:
        points = [(int(a), float(b)) for a, b in (p_.split(":") for p_ in args.sweep_points.split(","))]
    else:
        points = [(n, r) for n in (10_000, 100_000, 1_000_000, 10_000_000) for r in (0.1, 0.5, 1.0)]
        points += [(20_000_000, 0.5), (100_000_000, 0.5)]
    out = {"l2_bytes": l2, "copy_peak_gbs": hbm_peak, "points": [],
           "find_queries": "the activated keys in a fresh random order"}

    def timed(fn, reps=3, make=None):
        best = None
        for _ in range(reps):
            arg = make() if make else None
            flush.zero_()
            torch.cuda.synchronize()
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record()
            fn(arg)
            e1.record()
            torch.cuda.synchronize()
            ms = e0.elapsed_time(e1)
            best = ms if best is None else min(best, ms)
        return best

    clocks = ClockSampler(device.index)
    clocks.__enter__()
    t_start = time.time()
    for n, rho in points:
        keys = device_uniform_keys(n, rho, seed=1000 + n % 997 + int(rho * 10), device=device)
        g = torch.Generator(device=device)
        g.manual_seed(77 + n % 1000)
        queries = keys[torch.randperm(n, generator=g, device=device)].contiguous()
        holder = {}

        def make(tuning=None):
            holder["hm"] = ash.HashMap(3, n, device=device, tuning=tuning)
            torch.cuda.synchronize()
            return holder["hm"]

        with torch.cuda.nvtx.range(f"sweep_{n}_{rho}"):  # lets a profiler select one point
            ms_act = timed(lambda hm: hm.activate(keys), make=make)
            hm = holder["hm"]
            n_unique = hm.size()
            ms_find = timed(lambda _: hm.find(queries))
        small = small_call_figures(keys, queries, n, device, flush) if n <= 100_000 else None
        t = hm.tuning()
        slots = int(n * t.slots_per_capacity)
        ranged = 2 * slots * 8 > 3 * l2 and n >= (1 << 20)
        input_order = None
        if ranged:
            t1 = ash.default_tuning()
            t1.partition_keys = 1
            with torch.cuda.nvtx.range(f"sweep_input_order_{n}_{rho}"):
                io_act = timed(lambda hm_: hm_.activate(keys), make=lambda: make(t1))
                hm_io = holder["hm"]
                io_find = timed(lambda _: hm_io.find(queries))
            input_order = {"activate": io_act, "find": io_find}
            del hm_io
        # the random accesses touch one 32 B bucket per distinct key and its
        # 16 B kB row: a map of few distinct keys stays in L2 however large
        # its table is
        footprint = min(slots * 8, n_unique * 32) + min(n * 16, n_unique * 16)
        working = int(footprint + n * 12 + n * 5)   # + keys in, outputs
        rec = {"n": n, "rho": rho, "unique": n_unique, "working_set_x_l2": working / l2,
               "random_footprint_bytes": footprint}
        r_gbs = None
        if footprint >= l2:
            with torch.cuda.nvtx.range(f"probe_{n}_{rho}"):
                r_gbs, r_gsec = probe_random_gbs(footprint, device)
            rec["probe_random_read_gbs"] = r_gbs
            rec["probe_random_Gsectors"] = r_gsec
        splits = {"activate": split_activate(n, n_unique), "find": split_find(n, 0)}
        rec["ranged"] = ranged
        for name, ms in (("activate", ms_act), ("find", ms_find)):
            rnd, stm = splits[name]
            gbs = (rnd + stm) / (ms / 1000.0) / 1e9
            rec[name] = {"ms": ms, "keys_per_s": n / (ms / 1000.0), "algo_gbs": gbs, "frac_hbm": gbs / hbm_peak,
                         "random_bytes": rnd, "streamed_bytes": stm,
                         "random_Gsectors": rnd / 32 / (ms / 1000.0) / 1e9}
            if input_order is None:
                rec[name]["frac_random_access_roofline"] = random_access_fraction(ms, rnd, stm, r_gbs, hbm_peak)
            else:
                io = input_order[name]
                io_gbs = (rnd + stm) / (io / 1000.0) / 1e9
                rec[name]["speedup_vs_input_order"] = io / ms
                rec[name]["input_order"] = {
                    "ms": io, "keys_per_s": n / (io / 1000.0), "algo_gbs": io_gbs, "frac_hbm": io_gbs / hbm_peak,
                    "frac_random_access_roofline": random_access_fraction(io, rnd, stm, r_gbs, hbm_peak)}
        if small is not None:
            rec["per_call"] = small
        out["points"].append(rec)
        del hm, keys, queries
        holder.clear()
        torch.cuda.empty_cache()
    clocks.mark(t_start, time.time())
    clocks.__exit__(None, None, None)
    out["clocks"] = clocks.summary()
    return out


def tsdf_block_map_figures(args, device, hbm_peak):
    """The TSDF-shaped voxel-block map: 640x480 frames of synthetic smooth
    depth (6 mm voxels, 8^3 blocks, 48 mm block keys) along a slow path;
    capacity 2^20 with tsdf float32[8,8,8] and weight float16[8,8,8] value
    buffers.  Per frame the double hash map activates the frame's blocks
    (local map cleared per frame, global activate + find); after all frames
    the 27-neighbourhood of every active block is found.  Frame keys are on
    the device before timing."""
    import torch
    from paper_2110_00511_gb300 import ash, workloads
    frames = [torch.from_numpy(k).to(device) for k in workloads.tsdf_block_frames(n_frames=args.block_frames, seed=0)]
    n_points = sum(k.shape[0] for k in frames)
    stream = torch.cuda.current_stream(device)

    def run(trace):
        gmap = ash.HashMap(3, 1 << 20, [(8, 8, 8), (8, 8, 8)], [torch.float32, torch.float16], device=device)
        local = ash.HashMap(3, 1 << 19, [(1,)], [torch.int32], device=device)
        torch.cuda.synchronize()
        if trace:
            ash.ash_trace_reset()
            ash.ash_trace_enable(True)
        e0, e1, e2 = (torch.cuda.Event(enable_timing=True) for _ in range(3))
        e0.record(stream)
        n_unique = 0
        for k in frames:
            local.clear()
            uk, _, _ = ash.ash_double_map_activate(local, gmap, k)
            n_unique += uk.shape[0]
        e1.record(stream)
        act, cnt = gmap.active_indices_async()
        keys = gmap.gather_keys_count(act, cnt)
        n_blocks = int(cnt.item())
        e1b = torch.cuda.Event(enable_timing=True)
        e1b.record(stream)
        idx, mask = gmap.find_neighbors(keys[:n_blocks], 1)
        e2.record(stream)
        if trace:
            ash.ash_trace_enable(False)
        torch.cuda.synchronize()
        return (e0.elapsed_time(e1), e1b.elapsed_time(e2), n_unique, n_blocks, int(mask.sum().item()))

    run(False)  # warm-up: code, pools
    ms_frames, ms_nb, n_unique, n_blocks, n_hits = run(True)
    trace = ash.ash_trace_collect()
    kernels = {}
    tot = sum(t for t, n in trace.values())
    for name, (t, n) in trace.items():
        if n:
            kernels[name] = {"launches": n, "ms_per_launch": t / n, "share": t / tot if tot else 0.0}
    frame_ops = n_points + 2 * n_unique  # local activate + global activate and find
    nb = 27 * n_blocks
    nb_bytes = bytes_find(n_hits, nb - n_hits) - nb * 4 * 3 + n_blocks * 4 * 3  # keys read once per block
    return {"frames": len(frames), "points": n_points, "frame_unique_blocks": n_unique, "active_blocks": n_blocks,
            "ms_per_frame": ms_frames / len(frames),
            "frame_hash_ops_per_s": frame_ops / (ms_frames / 1000.0),
            "neighbourhood": {"queries": nb, "hits": n_hits, "ms": ms_nb, "ops_per_s": nb / (ms_nb / 1000.0),
                              "algo_gbs": nb_bytes / (ms_nb / 1000.0) / 1e9,
                              "frac_hbm": nb_bytes / (ms_nb / 1000.0) / 1e9 / hbm_peak},
            "kernels": kernels,
            "timing": "CUDA events; each frame synchronises once (the global map's growth check)"}


def bytes_integrate(n_blocks, n_updates, image_bytes):
    """Per listed block: its index (4) and kB row (16); per updated voxel: d
    and w read and written (16); the depth image read once (it stays in L2)."""
    return n_blocks * 20 + n_updates * 16 + image_bytes


def tsdf_figures(args, device, hbm_peak, with_cpu):
    """The voxel-block pipeline of Sec. 6.2 on 640x480 depth frames of a
    synthetic room: per frame depth -> block keys, the double hash map
    (local map cleared per frame), TSDF integration of the frame's blocks,
    and ray casting from the frame's pose through the local map.  6 mm voxels
    in 8^3 blocks, truncation 4 voxels, depth in (0, 4] m."""
    import torch
    from paper_2110_00511_gb300 import ash, workloads
    cam = workloads.Camera()
    voxel, ell = 0.006, 8
    trunc = 4 * voxel
    depth_max, depth_min = 4.0, 0.3
    step = voxel
    n_steps = int((depth_max - depth_min) / step)
    intr = (cam.fx, cam.fy, cam.cx, cam.cy)
    scene = workloads.room_scene(0)
    poses = workloads.camera_path(args.tsdf_frames, 0, turn=0.25)
    depths = [torch.from_numpy(workloads.render_depth(scene, ex, cam, noise=0.002, seed=j)).to(device)
              for j, ex in enumerate(poses)]
    local = ash.HashMap(3, 1 << 17, [(1,)], [torch.int32], device=device)
    vol = ash.HashMap(3, 1 << 19, [(ell, ell, ell), (ell, ell, ell)], [torch.float32, torch.float32], device=device)
    out = torch.empty((cam.height, cam.width), dtype=torch.float32, device=device)
    stream = torch.cuda.current_stream(device)

    def frame(j, trace_blocks):
        keys = ash.ash_depth_to_block_keys(depths[j], intr, poses[j], voxel * ell, depth_max)
        local.clear()
        _, _, gi = ash.ash_double_map_activate(local, vol, keys)
        ash.ash_tsdf_integrate(vol, gi, depths[j], intr, poses[j], voxel, trunc, depth_max)
        ash.ash_tsdf_raycast(vol, intr, poses[j], cam.width, cam.height, voxel, depth_min, step, n_steps,
                             local=local, out=out)
        trace_blocks.append(gi.numel())

    warm = []
    for j in range(min(3, len(poses))):
        frame(j, warm)
    torch.cuda.synchronize()
    # restart from an empty volume so the timed frames integrate the whole path
    vol = ash.HashMap(3, 1 << 19, [(ell, ell, ell), (ell, ell, ell)], [torch.float32, torch.float32], device=device)
    torch.cuda.synchronize()
    ash.ash_trace_reset()
    ash.ash_trace_enable(True)
    blocks = []
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record(stream)
    for j in range(len(poses)):
        frame(j, blocks)
    e1.record(stream)
    ash.ash_trace_enable(False)
    torch.cuda.synchronize()
    ms = e0.elapsed_time(e1)
    trace = ash.ash_trace_collect()
    n_updates = float(vol.value_buffer(1).sum().item())
    kernels = {}
    tot = sum(t for t, n in trace.values())
    for name, (t, n) in trace.items():
        if n:
            kernels[name] = {"launches": n, "ms_per_launch": t / n, "share": t / tot if tot else 0.0}
    integ_bytes = bytes_integrate(sum(blocks), n_updates, len(poses) * cam.width * cam.height * 4)
    res = {"frames": len(poses), "image": [cam.width, cam.height], "voxel_m": voxel, "block": ell,
           "trunc_m": trunc, "volume_blocks": vol.size(), "blocks_per_frame_mean": sum(blocks) / len(blocks),
           "ms_per_frame": ms / len(poses), "frames_per_s": 1000.0 * len(poses) / ms,
           "voxel_updates_per_frame": n_updates / len(poses), "kernels": kernels,
           "timing": "CUDA events around all frames; each frame synchronises twice (key count, new-key count)"}
    if "tsdf_integrate" in kernels:
        ki = kernels["tsdf_integrate"]
        gbs = integ_bytes / len(poses) / (ki["ms_per_launch"] / 1000.0) / 1e9
        res["integrate"] = {"algo_bytes_per_frame": integ_bytes / len(poses), "achieved_gbs": gbs,
                            "frac_hbm": gbs / hbm_peak,
                            "voxels_per_s": sum(blocks) * ell ** 3 / (ki["ms_per_launch"] * len(poses) / 1000.0)}
    if "tsdf_raycast" in kernels:
        kr = kernels["tsdf_raycast"]
        res["raycast"] = {"rays_per_s": cam.width * cam.height / (kr["ms_per_launch"] / 1000.0),
                          "ns_per_ray": kr["ms_per_launch"] * 1e6 / (cam.width * cam.height),
                          "max_samples_per_ray": n_steps, "through": "the frame's local map"}
    # the double-hash-map speed-up of Sec. 6.2: the same ray casting through
    # the whole volume's map and through the last frame's local map
    def timed_rc(use_local, reps=5):
        best = None
        for _ in range(reps):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record(stream)
            ash.ash_tsdf_raycast(vol, intr, poses[-1], cam.width, cam.height, voxel, depth_min, step, n_steps,
                                 local=local if use_local else None, out=out)
            b.record(stream)
            torch.cuda.synchronize()
            best = a.elapsed_time(b) if best is None else min(best, a.elapsed_time(b))
        return best
    ms_global, ms_local = timed_rc(False), timed_rc(True)
    res["raycast_global_vs_local"] = {"ms_global_map": ms_global, "ms_local_map": ms_local,
                                      "speedup": ms_global / ms_local if ms_local else None}
    # inputs for the CPU oracle's timing of one frame (run by the cpu_baseline leg)
    cpu_inputs = {"depth": depths[0].cpu().numpy(), "pose": poses[0], "intr": intr, "cam": cam, "voxel": voxel,
                  "ell": ell, "trunc": trunc, "depth_max": depth_max, "depth_min": depth_min, "step": step,
                  "n_steps": n_steps} if with_cpu else None
    return res, cpu_inputs


def per_op_figures(args, device, hbm_peak):
    """Per-op throughput at the uniform 10^7-key point (rho = 0.5), whose
    table and key buffer exceed L2: insert, find (hits), find (misses), erase,
    activate and rehash, each timed with CUDA events, L2 flushed before each."""
    import torch
    from paper_2110_00511_gb300 import ash, workloads
    n = args.ops_n
    keys_np = workloads.uniform_keys(n, 0.5, seed=11)
    keys = torch.from_numpy(keys_np).to(device)
    miss = keys + (1 << 21)  # outside the generator's [-2^20, 2^20) range: all absent
    vals = torch.rand(n, device=device)
    flush = torch.empty(L2_FLUSH_BYTES, dtype=torch.uint8, device=device)
    n_unique = int(round(0.5 * n))
    out = {"n": n, "rho": 0.5, "unique": n_unique}

    def timed(fn, reps=3):
        best = None
        for _ in range(reps):
            flush.zero_()
            torch.cuda.synchronize()
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record()
            fn()
            e1.record()
            torch.cuda.synchronize()
            ms = e0.elapsed_time(e1)
            best = ms if best is None else min(best, ms)
        return best

    def rec(name, ms, nbytes, nops):
        gbs = nbytes / (ms / 1000) / 1e9
        out[name] = {"ms": ms, "ops_per_s": nops / (ms / 1000), "algo_gbs": gbs, "frac_hbm": gbs / hbm_peak}

    state = {}

    def do_insert():
        state["hm"] = ash.HashMap(3, n, [(1,)], [torch.float32], device=device)
        torch.cuda.synchronize()
        return None

    # insert timed without map creation
    ms_ins = []
    for _ in range(3):
        do_insert()
        flush.zero_()
        torch.cuda.synchronize()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        state["hm"].insert(keys, [vals])
        e1.record()
        torch.cuda.synchronize()
        ms_ins.append(e0.elapsed_time(e1))
    hm = state["hm"]
    t = hm.tuning()
    rec("insert", min(ms_ins), bytes_claim(n) + bytes_commit(n, n_unique, 4), n)
    rec("find_hit", timed(lambda: hm.find(keys)), bytes_find(n, 0), n)
    rec("find_miss", timed(lambda: hm.find(miss)), bytes_find(0, n), n)
    # thread-per-key vs warp-cooperative probing, on 32 B and 128 B buckets
    cmp = {}
    for S in (4, 16):
        tt = ash.default_tuning()
        tt.slots_per_bucket = S
        hp = ash.HashMap(3, n, device=device, tuning=tt)
        hp.activate(keys)
        for wp in (0, 1):
            tt.warp_probe = wp
            hp.set_tuning(tt)
            name = f"S{S}_{'warp_group' if wp else 'thread_per_key'}"
            ms_h = timed(lambda: hp.find(keys))
            ms_m = timed(lambda: hp.find(miss))
            cmp[name] = {"find_hit_ops_per_s": n / (ms_h / 1000), "find_miss_ops_per_s": n / (ms_m / 1000)}
        del hp
    out["probe_compare"] = cmp
    ms_act = []
    for _ in range(3):
        h2 = ash.HashMap(3, n, device=device)
        flush.zero_()
        torch.cuda.synchronize()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        h2.activate(keys)
        e1.record()
        torch.cuda.synchronize()
        ms_act.append(e0.elapsed_time(e1))
        del h2
    rec("activate", min(ms_act), bytes_claim(n) + bytes_commit(n, n_unique, 0), n)
    import math
    n_slots = int(math.ceil(n * t.slots_per_capacity / t.slots_per_bucket)) * t.slots_per_bucket
    rec("list_active", timed(lambda: hm.active_indices()), bytes_list(n, n_unique), n_unique)
    ms_er = []
    for _ in range(2):
        h3 = ash.HashMap(3, n, device=device)
        h3.activate(keys)
        flush.zero_()
        torch.cuda.synchronize()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        h3.erase(keys)
        e1.record()
        torch.cuda.synchronize()
        ms_er.append(e0.elapsed_time(e1))
        del h3
    rec("erase", min(ms_er), bytes_erase(n_unique, 0) + (n - n_unique) * (4 * 3 + 5 + 64), n)
    ms_rh = timed(lambda: hm.rehash(2 * hm.capacity()), reps=1)
    c = hm.capacity() // 2
    n_slots2 = 2 * n_slots
    rh_bytes = bytes_list(c, n_unique) + 8 * n_slots2 + n_unique * (4 + 16 + 64) + 2 * c * (16 + 4 + 4)
    rec("rehash_x2", ms_rh, rh_bytes, n_unique)
    del hm
    return out


def batched_figures(args, device, reps=15):
    """Many maps, one mixed batch each (key_dim 2-4, capacities log-uniform in
    2^10..2^21, 30/60/10 insert/find/erase, rho ~ U(0.2, 1)), serviced (a) as
    ONE run of the batched kernels and (b) as plain per-map calls
    (insert, find, erase for each map) through the same binding.  Maps are
    cleared between repetitions (untimed); each repetition is timed with CUDA
    events around the whole service."""
    import torch
    from paper_2110_00511_gb300 import ash, workloads
    cases = workloads.batched_maps(n_maps=args.batched_maps, seed=0)
    tunings = [ash.ash_autotune(c.key_dim, c.capacity, c.rho, device.index) for c in cases]
    dev_data = [(torch.from_numpy(c.insert_keys).to(device), torch.from_numpy(c.insert_values).to(device),
                 torch.from_numpy(c.find_keys).to(device), torch.from_numpy(c.erase_keys).to(device)) for c in cases]
    n_ops = sum(len(c.insert_keys) + len(c.find_keys) + len(c.erase_keys) for c in cases)

    def make_maps():
        return [ash.HashMap(c.key_dim, c.capacity, [(1,)], [torch.float32], device=device, tuning=t)
                for c, t in zip(cases, tunings)]

    maps_b, maps_p = make_maps(), make_maps()
    batch = ash.Batch(device.index)
    items = []
    outputs = []
    for hm, (ik, iv, fk, ek) in zip(maps_b, dev_data):
        items += [(hm, ash.ASH_OP_INSERT, ik, iv), (hm, ash.ASH_OP_FIND, fk, None), (hm, ash.ASH_OP_ERASE, ek, None)]
        outputs += [(torch.empty(len(ik), dtype=torch.int32, device=device), torch.empty(len(ik), dtype=torch.bool, device=device)),
                    (torch.empty(len(fk), dtype=torch.int32, device=device), torch.empty(len(fk), dtype=torch.bool, device=device)),
                    (None, torch.empty(len(ek), dtype=torch.bool, device=device))]

    def run_batched():
        batch.run(items, outputs)

    def run_plain():
        for hm, (ik, iv, fk, ek) in zip(maps_p, dev_data):
            hm.insert(ik, [iv])
            hm.find(fk)
            hm.erase(ek)

    res = {}
    for name, fn, maps in (("batched_graph", run_batched, maps_b), ("plain_per_map", run_plain, maps_p)):
        times = []
        for r in range(reps + 2):
            for hm in maps:
                hm.clear()
            torch.cuda.synchronize()
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record()
            fn()
            e1.record()
            torch.cuda.synchronize()
            if r >= 2:
                times.append(e0.elapsed_time(e1))
        times_sorted = sorted(times)
        res[name] = {"ms_median": statistics.median(times),
                     "ms_p99": times_sorted[min(len(times) - 1, int(0.99 * len(times)))],
                     "ops_per_s": n_ops / (statistics.median(times) / 1000.0)}
    res["maps"] = len(cases)
    res["ops_per_batch"] = n_ops
    res["speedup_ops_per_s"] = res["batched_graph"]["ops_per_s"] / res["plain_per_map"]["ops_per_s"]
    res["timing"] = ("CUDA events on the stream around the whole service of all maps' batches (the plain "
                     "form's span includes GPU idle time while the host issues its calls)")
    return res


def _pct(xs, q):
    xs = sorted(xs)
    return xs[min(len(xs) - 1, int(q * len(xs)))] if xs else None


def serving_figures(args, device, n_tenants=16, clients=8):
    """Poisson arrivals over 16 resident tenant maps (int32x3 keys, one f32
    value), request sizes log-uniform in 1e3..1e6 keys, ops 30/60/10
    insert/find/erase; request keys and values in pinned host memory.  Every
    form replays the same traces from native threads (ash_server_replay /
    ash_replay_sequential), so the client side adds no interpreter time:
      served             the continuous-batching server, mode 0 (keys copied
                         into pinned staging at submit);
      served_pinned_dma  mode 2 (pinned request arrays uploaded by DMA, no
                         CPU copy): the recommended form for callers whose
                         request buffers are pinned, which is the case here;
      served_zero_copy   mode 1 (kernels use the callers' arrays in place),
                         where the device reads pageable host memory;
      sequential_plain   the same requests as plain calls in arrival order
                         (upload, op, download, synchronise).
    Latency = outputs in the caller's arrays - scheduled arrival.  Each rate
    runs `repeats` traces of `requests` requests; per form the median over
    repeats is reported with the spread (min, max) of p50, p99 and req/s.
    p99.9 is reported only when at least 1000 requests lie beyond it."""
    import torch
    from paper_2110_00511_gb300 import ash
    rng = np.random.default_rng(5)
    pool_n = 8_000_000
    key_pool = torch.from_numpy(rng.integers(-(1 << 18), 1 << 18, size=(pool_n, 3)).astype(np.int32)).pin_memory()
    val_pool = torch.from_numpy(rng.random(pool_n, dtype=np.float32)).pin_memory()
    keys_np, vals_np = key_pool.numpy(), val_pool.numpy()
    ops_of = np.array([ash.ASH_OP_INSERT, ash.ASH_OP_FIND, ash.ASH_OP_ERASE])
    rates = [float(x) for x in args.serving_rates.split(",") if x]
    R, reps = args.serving_requests, args.serving_repeats
    zc = ash.ash_get_device_info(device.index)["pageable_memory_access"] == 1
    out = {"tenants": n_tenants, "requests_per_trace": R, "repeats": reps, "client_threads": clients,
           "default_mode": "served_zero_copy" if zc else "served_pinned_dma",
           "default_mode_reason": "on a coherent CPU-GPU node mode 1 (kernels read the request arrays in place) "
                                  "has the lowest latency and the highest throughput at every rate; elsewhere mode 2 "
                                  "(DMA from the pinned request arrays); the server's API default stays mode 0, "
                                  "the only mode whose callers may reuse their arrays as soon as submit returns",
           "client": "native replay threads (no interpreter in the measured path)", "rates": {}}

    def make_trace(rate, seed):
        g = np.random.default_rng(seed)
        arr = np.cumsum(g.exponential(1.0 / rate, size=R))
        sizes = np.exp(g.uniform(np.log(1e3), np.log(1e6), size=R)).astype(np.int64)
        ops = ops_of[g.choice(3, size=R, p=[0.3, 0.6, 0.1])]
        tenants = g.integers(0, n_tenants, size=R)
        starts = g.integers(0, pool_n - sizes)
        return ash.Trace(arr, tenants, ops, sizes, starts, keys_np, vals_np)

    def summarize(lat_ms, keys_total, span_s):
        lat = np.sort(np.asarray(lat_ms))
        rec = {"p50_ms": float(np.percentile(lat, 50)), "p99_ms": float(np.percentile(lat, 99)),
               "req_per_s": len(lat) / span_s, "keys_per_s": keys_total / span_s}
        if len(lat) * 0.001 >= 1000:
            rec["p999_ms"] = float(np.percentile(lat, 99.9))
        return rec

    def mk(mode):
        return ash.Server(n_tenants=n_tenants, key_dim=3, initial_capacity=1 << 20, value_row_bytes=4,
                          device=device.index, staging_bytes=4 << 30, max_load=0.7, max_batch_requests=256,
                          zero_copy=mode)

    forms = {"served": mk(0), "served_pinned_dma": mk(2)}
    if zc:
        forms["served_zero_copy"] = mk(1)
    maps = [ash.HashMap(3, 1 << 20, [(1,)], [torch.float32], device=device) for _ in range(n_tenants)]
    warm = make_trace(2000.0, 99)
    warm.n_requests = min(warm.n_requests, 400)
    for name, srv in forms.items():
        srv.replay(warm, clients)
    ash.replay_sequential(maps, warm)

    for ri, rate in enumerate(rates):
        runs = {k: [] for k in list(forms) + ["sequential_plain"]}
        batches = {k: [0, 0, 0, 0, 0] for k in forms}
        offered = []
        for rep in range(reps):
            tr = make_trace(rate, 100 + 10 * ri + rep)
            keys_total = int(tr.n.sum())
            offered.append(keys_total / float(tr.arrival_s[-1]))
            for name, srv in forms.items():
                st0 = srv.stats()
                lat, span = srv.replay(tr, clients)
                st1 = srv.stats()
                runs[name].append(summarize(lat, keys_total, span))
                print(f"serving {int(rate)} rep {rep} {name}: {len(lat) / span:.0f} req/s p99 "
                      f"{np.percentile(lat, 99):.2f} ms", file=sys.stderr, flush=True)
                batches[name][0] += st1["batches"] - st0["batches"]
                batches[name][1] += st1["batched_requests"] - st0["batched_requests"]
                batches[name][2] += st1["rehashes"] - st0["rehashes"]
                batches[name][3] += st1["host_syncs"] - st0["host_syncs"]
                batches[name][4] += st1["pinned_spills"] - st0["pinned_spills"]
            lat, span = ash.replay_sequential(maps, tr)
            runs["sequential_plain"].append(summarize(lat, keys_total, span))
        entry = {"offered_keys_per_s": float(np.median(offered))}
        for name, recs in runs.items():
            agg = {}
            for k in recs[0]:
                vals = [r_[k] for r_ in recs]
                agg[k] = float(np.median(vals))
                agg[k + "_range"] = [float(min(vals)), float(max(vals))]
            if name in batches:
                nb, nr, nrh, nsync, nspill = batches[name]
                agg["avg_requests_per_batch"] = nr / max(1, nb)
                agg["growth_rehashes"] = nrh
                agg["host_syncs"] = nsync
                agg["pinned_spills"] = nspill
            entry[name] = agg
        out["rates"][str(int(rate))] = entry
    for srv in forms.values():
        srv.close()
    del maps
    return out


if __name__ == "__main__":
    sys.exit(main())
