"""Voxel claims from the leaf upwards: grids and sides around the point where a
cell is one unit wide, leaves of one point, unsplittable leaves of equal
points, batches around a warp, re-inserted points of several levels, and a
restored octree whose voxels do not nest. Compared with the oracle's closed
form byte for byte."""
import numpy as np
import pytest

import oracle
from helpers import assert_snapshots_equal
from paper_2310_03567_gb300 import simlod, synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def make(root, T, C, G, n):
    kw = dict(root_log2=root, leaf_capacity=T, chunk_points=C, grid_log2=G)
    cfg = simlod.default_config(max_batch_points=1 << 18, spill_capacity=1 << 20,
                                backlog_capacity=1 << 22, max_nodes=1 << 19, **kw)
    tree = simlod.Octree(cfg, simlod.make_arena(cfg, 3 << 30), stream=torch.cuda.Stream())
    return tree, oracle.Config.make(**kw)


def points(kind, root, n):
    if kind == "uniform":
        return synth.uniform(11, 1 << root, n)
    rng = np.random.default_rng(5)
    p = synth.uniform(12, 1 << root, n)
    if kind == "dense":  # most points in one corner, many of them equal
        for f in "xyz":
            p[f][: n - n // 8] = rng.integers(0, max(2, 1 << max(0, root - 6)), n - n // 8)
    return p


@pytest.mark.parametrize("root,G", [(3, 7), (5, 3), (7, 7), (9, 2), (16, 7), (20, 6)])
@pytest.mark.parametrize("kind", ["uniform", "dense"])
@pytest.mark.parametrize("T,C,cuts", [(1, 1, (31, 1, 33, 500)), (40, 7, (32, 2_000, 65, 4_000)),
                                      (700, 100, (9_000, 1, 20_000))])
def test_claims_match_the_closed_form(root, G, kind, T, C, cuts):
    n = sum(cuts)
    pts = points(kind, root, n)
    tree, ocfg = make(root, T, C, G, n)
    cut = np.split(pts, np.cumsum(cuts)[:-1])
    for form in ("fused", "plain"):
        tree.reset()
        if form == "fused":
            tree.insert_many([simlod.points_tensor(b) for b in cut])
        else:
            for b in cut:
                tree.insert(simlod.points_tensor(b))
        assert tree.sync() == simlod.OK
        assert_snapshots_equal(tree.snapshot(), oracle.static_build(ocfg, pts))


def test_restored_voxels_that_do_not_nest_are_claimed_cell_by_cell():
    # half of the root's voxels are missing from the checkpoint although the
    # nodes below hold the same places: later points fill exactly the gaps
    pts = synth.uniform(3, 1 << 14, 30_000)
    tree, ocfg = make(14, 4_000, 64, 5, 60_000)
    tree.insert_many([simlod.points_tensor(pts)])
    snap = tree.snapshot()
    assert snap.nodes["is_inner"][0] and snap.nodes["is_inner"].sum() == 1
    more = pts[::7].copy()  # the same places again, in other colours
    for f in "rgba":
        more[f] ^= 0x5A
    gone = np.arange(len(snap.voxels)) % 2 == 0
    broken = simlod.Snapshot(snap.nodes.copy(), snap.points, snap.voxels[~gone])
    broken.nodes["n_voxels"][0] = (~gone).sum()
    broken.nodes["n_chunks"][0] = -(-int((~gone).sum()) // 64)
    other, _ = make(14, 4_000, 64, 5, 60_000)
    for form in ("fused", "plain"):
        other.restore(broken)
        if form == "fused":
            other.insert_many([simlod.points_tensor(more)])
        else:
            other.insert(simlod.points_tensor(more))
        assert other.sync() == simlod.OK
        got = other.snapshot()
        # the leaf points of the checkpoint lie in the missing cells as well,
        # but they sampled the root when they came: only `more` makes voxels
        cells = ((more["x"] >> 9).astype(np.int64) | ((more["y"] >> 9).astype(np.int64) << 5) |
                 ((more["z"] >> 9).astype(np.int64) << 10))
        first = {}
        for k, cell in enumerate(cells):
            first.setdefault(int(cell), k)
        have = {int(v["cell"]): int(v["rgba"]) for v in broken.voxels}
        for cell, k in first.items():
            p = more[k]
            have.setdefault(cell, int(p["r"]) | int(p["g"]) << 8 | int(p["b"]) << 16 |
                            int(p["a"]) << 24)
        root = {int(v["cell"]): int(v["rgba"]) for v in got.voxels[:int(got.nodes["n_voxels"][0])]}
        assert root == have
        assert len(got.points) == len(pts) + len(more)
