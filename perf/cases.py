"""What a user of this framework has it do, as cases that can be timed.

A case names a point stream (which scan-like distribution, how many points,
how they are cut into batches) and the form in which a program hands it to the
octree: packet by packet, batch by batch (plain form), one persistent launch
over many batches (fused form), a plan that merges uneven batches (batched
form), pinned host batches (host-fed form), two octrees side by side, frames
of a finished octree, compaction, or a checkpoint. Every pass that builds an
octree starts from an empty one, ends with what a program reads back (status
and counters) and draws a frame with a camera inside the scene, so that points
of near leaves and voxels of every coarser level are in it.

All outputs are whole numbers: frames are 64-bit words (depth bits << 32 |
rgba), counters are integers, snapshots are records. They are compared word by
word, so there is no 64-bit result to measure a rounding against.
"""
import math

import numpy as np
import torch

from paper_2310_03567_gb300 import simlod, synth

# New voxels per inserted point of the streams (measured on this library's
# counters at a few million points and more; used for byte counts only).
VOXELS_PER_POINT = {"uniform": 1.5, "aerial": 0.42, "clustered": 0.13, "morton": 0.13,
                    "mixed": 0.3}
COUNTERS = ("batches", "points", "rejected_batches", "spilled", "splits", "voxels",
            "iterations_max", "nodes")


def listed():
    def case(name, form, kind, n, lo, hi=None, width=1920, height=1080, chunk=1000,
             views=1):
        return {"name": name, "form": form, "kind": kind, "n": n, "batch_lo": lo,
                "batch_hi": hi or lo, "width": width, "height": height, "chunk": chunk,
                "views": views}

    return [
        # a scanner's packets as they arrive, one launch each, then the frame:
        # launches and waits count
        case("packets-64k", "packets", "aerial", 65_536, 4_096, width=1280, height=720),
        # the plain form on the paper-style uniform stream of 100k batches
        case("plain-uniform-1M", "plain", "uniform", 1_000_000, 100_000),
        # the plain form with ragged batches and small chunks
        case("plain-clustered-5M", "plain", "clustered", 5_234_567, 77_777, 1_500_000, chunk=500),
        # an aerial scan in scan-line order, 1M-point batches, one launch
        case("fused-aerial-16M", "fused", "aerial", 16_000_000, 1_000_000),
        # a building scan, 1M-10M batches in shuffled order, one launch, drawn
        # from near and from above
        case("fused-clustered-120M", "fused", "clustered", 120_000_000, 1_000_000, 10_000_000,
             3840, 2160, views=2),
        # the same kind of scan sorted along the z-curve
        case("fused-morton-6M", "fused", "morton", 6_000_000, 1_000_000),
        # uneven batches, 64k to 8M, merged by a plan that is kept
        case("plan-mixed-24M", "plan", "mixed", 24_000_000, 65_536, 8_388_608, views=2),
        # pinned host batches of an odd size, copies beside the updates
        case("hostfed-aerial-6M", "hostfed", "aerial", 6_250_001, 617_283),
        # a server's two octrees, half the GPU each, at the same time
        case("pair-clustered-4M", "pair", "clustered", 4_000_000, 250_000, 1_000_000),
        # frames of a finished terrain: an overview and a close view
        case("frames-aerial-12M", "frames", "aerial", 12_000_000, 1_000_000, views=2),
        # an octree built, its cold nodes turned into arrays, and drawn
        case("compact-clustered-12M", "compact", "clustered", 12_000_000, 500_000, 3_000_000),
        # a checkpoint (the whole octree, record by record) written and read back
        case("checkpoint-mixed-2M", "checkpoint", "mixed", 2_000_003, 65_536, 1_048_576),
    ]


def draw(rng):
    form = rng.choice(["packets", "plain", "plain", "fused", "fused", "fused", "plan", "hostfed",
                       "pair", "frames", "compact", "checkpoint"])
    kinds = ["uniform", "aerial", "clustered", "mixed", "clustered", "aerial"]
    if form in ("plain", "fused"):
        kinds.append("morton")
    kind = rng.choice(kinds)
    lo, hi = {"packets": (20_000, 1_000_000), "plain": (50_000, 16_000_000),
              "fused": (50_000, 48_000_000), "plan": (200_000, 24_000_000),
              "hostfed": (50_000, 16_000_000), "pair": (50_000, 8_000_000),
              "frames": (50_000, 16_000_000), "compact": (200_000, 16_000_000),
              "checkpoint": (20_000, 3_000_000)}[form]
    if kind == "uniform":
        hi = min(hi, 12_000_000)
    if kind == "morton":
        hi = min(hi, 8_000_000)
    if kind == "uniform" and form == "checkpoint":
        hi = 1_000_000
    n = int(math.exp(rng.uniform(math.log(lo), math.log(hi))))
    least = max(1_000, n // 24 if form == "packets" else n // 64)
    b_lo = int(math.exp(rng.uniform(math.log(least), math.log(max(least + 1, min(n, 4_000_000))))))
    b_hi = b_lo if rng.random() < 0.4 else min(8_388_608, int(b_lo * rng.uniform(1.2, 12)))
    width, height = rng.choice([(640, 480), (1280, 720), (1366, 768), (1920, 1080), (3840, 2160)])
    return {"form": form, "kind": kind, "n": n, "batch_lo": b_lo, "batch_hi": b_hi,
            "width": width, "height": height,
            "chunk": rng.choice([250, 500, 1000, 1000, 1000, 2000, 5000]),
            "views": rng.choice([1, 2])}


def _quads(n):
    """Quads of a clustered scan of n points (15,000 points per quad)."""
    return max(8, n // 15_000)


def _stream(case, seed):
    """(points in insertion order, batch counts, root_log2)."""
    kind, n = case["kind"], case["n"]
    if kind == "uniform":
        pts, root = synth.uniform(seed, 1_000_000, n), 20
    elif kind == "aerial":
        pts, root = synth.terrain(seed, n), 22
    elif kind == "mixed":
        w = synth.mixed_workload(n, seed, run_lo=max(1, n // 40), run_hi=max(2, n // 10))
        pts, root = w.points, 22
    else:
        pts, root = synth.clustered(seed, _quads(n), n), 21
    lo, hi = case["batch_lo"], max(case["batch_lo"], case["batch_hi"])
    if case["form"] == "plan" and hi > lo:
        off, cnt = synth.batch_cut_loguniform(seed, n, lo, hi)
    else:
        off, cnt = synth.batch_cut(seed, n, lo, hi, permute=kind == "clustered" and hi > lo)
    off, cnt = off.astype(np.int64), cnt.astype(np.int64)
    w = synth.Workload(kind, pts, off, cnt, (0, 0, 0), root, "")
    if kind == "morton":
        w = synth.morton_workload(w)
    return w.stream(), [int(c) for c in cnt], root


def _config(case, root, largest, merged):
    # an update re-inserts at most the whole octree; a uniform one whose leaves
    # all split at once makes a voxel for nearly every point of it
    most = max(merged, largest)
    voxels = 2 * case["n"] + (1 << 20)
    return simlod.default_config(
        root_log2=root, chunk_points=case["chunk"], max_batch_points=most,
        spill_capacity=max(8 << 20, case["n"]), max_nodes=1 << 19,
        backlog_capacity=min(voxels, (32 if case["kind"] == "uniform" else 16) << 20))


def _octree(case, cfg, stream=None):
    n = case["n"]
    v = 2.0 if case["kind"] == "uniform" else 0.8
    data = int(n * 20 * (1 + v) * 1.5) + (512 << 20) + 40_000 * 20 * case["chunk"] // 10
    data += (n // 6_000 + 64) * 300_000  # grids and directories
    return simlod.Octree(cfg, simlod.make_arena(cfg, data), stream=stream)


def _split(buf, counts):
    out, at = [], 0
    for c in counts:
        out.append(buf[at:at + c])
        at += c
    return out


def _cameras(pts, aspect):
    """A close view along the ground from inside the scene, and an overview."""
    step = max(1, len(pts) // 100_000)
    xyz = np.stack([pts[f][::step].astype(np.float64) for f in "xyz"], 1)
    lo, hi = xyz.min(0), xyz.max(0)
    ext = np.maximum(hi - lo, 1.0)
    ctr = (lo + hi) / 2
    side = ext.max()
    near = lo + ext * np.array([0.3, 0.3, 0.0])
    near[2] = hi[2] + 0.01 * side
    return [simlod.view_proj(near, ctr, 60.0, aspect),
            simlod.view_proj(ctr + side * np.array([-0.45, -0.55, 0.5]), ctr, 60.0, aspect)]


def prepare(case, seed):
    form = case["form"]
    pts, counts, root = _stream(case, seed)
    n, largest = len(pts), max(counts)
    merged = min(8_388_608, n) if form == "plan" else 0
    cfg = _config(case, root, largest, merged)
    frames = [torch.empty((case["height"], case["width"]), dtype=torch.int64, device="cuda")
              for _ in range(2)]
    views = case["views"]
    st = {"form": form, "cams": _cameras(pts, case["width"] / case["height"])[:views],
          "frames": frames[:2 if form == "pair" else views]}
    records = pts.view(np.uint8).reshape(-1, 16)
    if form == "hostfed":
        host = torch.empty((n, 16), dtype=torch.uint8, pin_memory=True)
        host.numpy()[:] = records
        st["host"] = _split(host, counts)
        st["dst"] = torch.empty((n, 16), dtype=torch.uint8, device="cuda")
        st["ready"] = torch.zeros(len(counts), dtype=torch.int32, device="cuda")
        st["copy"] = torch.cuda.Stream()
    else:
        st["batches"] = _split(torch.from_numpy(records).cuda(), counts)
    if form == "pair":
        st["trees"] = []
        for k in range(2):
            s = torch.cuda.Stream()
            tree = _octree(case, cfg, s)
            tree.set_launch_width(1)
            st["trees"].append(tree)
        return st
    tree = st["tree"] = _octree(case, cfg)
    if form == "plan":
        st["plan"] = tree.plan([b.data_ptr() for b in st["batches"]], counts, merge_points=merged)
    if form in ("frames", "checkpoint"):
        tree.insert_many(st["batches"])
        if tree.sync() != simlod.OK:
            raise RuntimeError("the octree was not built")
        del st["batches"]
    if form == "checkpoint":
        st["other"] = _octree(case, cfg)
        # room for the records of any octree of this size
        st["room"] = [np.zeros((k, w), np.int32) for k, w in
                      ((n // 500 + 1_024, 12), (n, 5), (4 * n + 4_096, 5))]
    return st


def _counters(tree, more=()):
    s = tree.stats()
    return [s[k] for k in COUNTERS + tuple(more)]


def _draw(tree, cams, frames):
    for cam, frame in zip(cams, frames):
        tree.render(cam, frame)


def run(state):
    form, frames, cams = state["form"], state["frames"], state["cams"]
    if form == "pair":
        # both octrees update at once; the caller's stream then takes the frames
        for tree in state["trees"]:
            tree.reset()
        half = len(state["batches"]) // 2
        shares = (state["batches"][:half], state["batches"][half:])
        for tree, share in zip(state["trees"], shares):
            tree.insert_many(share)
        for tree, frame in zip(state["trees"], frames):
            tree.render(cams[0], frame)
            torch.cuda.current_stream().wait_stream(tree.stream)
        return [frames] + [_counters(t) for t in state["trees"]]
    tree = state["tree"]
    if form == "frames":
        _draw(tree, cams, frames)
        return frames
    if form == "checkpoint":
        snap = tree.snapshot()
        state["other"].restore(snap)
        _draw(state["other"], cams, frames)
        for room, records in zip(state["room"], (snap.nodes, snap.points, snap.voxels)):
            room[:len(records)] = records.view(np.int32).reshape(len(records), -1)
        return [frames, len(snap.nodes), len(snap.points), len(snap.voxels)] + state["room"]
    tree.reset()
    if form == "packets":
        for b in state["batches"]:
            tree.insert_many([b])
        _draw(tree, cams, frames)
        return frames
    more = ()
    if form == "plain":
        for b in state["batches"]:
            tree.insert(b)
    elif form == "plan":
        state["plan"].run()
    elif form == "hostfed":
        tree.insert_many_host(state["host"], state["dst"], state["ready"], state["copy"])
    else:
        tree.insert_many(state["batches"])
    if form == "compact":
        tree.compact()
        more = ("compact_nodes", "compact_chunks", "compact_chunks_freed")
    _draw(tree, cams, frames)
    return [frames, tree.sync(), _counters(tree, more)]


def exact(case, seed):
    """Every output is a whole number."""
    return None


def work(case):
    """Points read (16 bytes), stored (20 bytes with their index), voxels
    stored (20 bytes with their cell), frame words written."""
    n, form = case["n"], case["form"]
    voxels = VOXELS_PER_POINT[case["kind"]] * n
    pixels = case["width"] * case["height"] * (2 if form == "pair" else case["views"])
    frame = 8 * pixels
    if form == "frames":
        # at least one record read for every pixel that shows one
        return {"bytes": frame + 16 * min(case["views"] * n, pixels // 2), "flops": 0}
    if form == "checkpoint":
        # records read, written as a snapshot, read and written as an octree
        return {"bytes": 80 * (n + voxels) + frame, "flops": 0}
    total = 36 * n + 20 * voxels + frame
    if form == "compact":
        total += 40 * (n + voxels)
    return {"bytes": total, "flops": 0}
