"""Batch lists around the length that travels in the launch itself (16), launch
after launch on one handle, with an empty batch and a rejected one among them,
and after a launch that was aborted: the control words clear themselves."""
import numpy as np
import pytest

import oracle
from helpers import assert_snapshots_equal
from paper_2310_03567_gb300 import simlod, synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

KW = dict(root_log2=16, leaf_capacity=300, chunk_points=40, grid_log2=5)


def make():
    cfg = simlod.default_config(max_batch_points=1 << 16, spill_capacity=1 << 18,
                                backlog_capacity=1 << 19, max_nodes=1 << 15, **KW)
    return simlod.Octree(cfg, simlod.make_arena(cfg, 256 << 20), stream=torch.cuda.Stream())


@pytest.mark.parametrize("lists", [(1, 16, 17), (15, 1, 1), (40, 16)])
def test_lists_of_any_length(lists):
    tree, kept, lo = make(), [], 0
    pts = synth.uniform(8, 1 << 16, 40_000)
    out = pts[:10].copy()
    out["y"][3] = 1 << 16  # outside the root cube: the batch is rejected whole
    for n in lists:
        batches = []
        for k in range(n):
            size = 0 if k % 7 == 3 else 33 + 11 * k
            batches.append(pts[lo:lo + size])
            kept.append(batches[-1])
            lo += size
        ts = [simlod.points_tensor(b) for b in batches]
        ts.insert(n // 2, simlod.points_tensor(out))
        tree.insert_many(ts)
        assert tree.sync() == simlod.ERR_OUT_OF_BOUNDS
    want = oracle.static_build(oracle.Config.make(**KW), np.concatenate(kept))
    assert_snapshots_equal(tree.snapshot(), want)


@pytest.mark.parametrize("synced", [True, False])
def test_a_launch_after_an_aborted_one(synced):
    # too many nodes: the first launch ends early with its blocks at different
    # barriers; the reset (with and without the status having been read) and
    # the next launch start clean
    pts = synth.uniform(9, 1 << 16, 60_000)
    cfg = simlod.default_config(max_batch_points=1 << 16, spill_capacity=1 << 18,
                                backlog_capacity=1 << 19, max_nodes=400, **KW)
    tree = simlod.Octree(cfg, simlod.make_arena(cfg, 256 << 20), stream=torch.cuda.Stream())
    ts = [simlod.points_tensor(pts[k:k + 3_000]) for k in range(0, len(pts), 3_000)]
    tree.insert_many(ts)
    if synced:
        assert tree.sync() == simlod.ERR_NODES_FULL
    tree.reset()
    tree.insert_many(ts[:2])
    assert tree.sync() == simlod.OK
    want = oracle.static_build(oracle.Config.make(**KW), pts[:6_000])
    assert_snapshots_equal(tree.snapshot(), want)


@pytest.mark.parametrize("sizes", [(0, 0, 3_000, 0, 0, 0, 5_000, 0), (0,) * 20 + (4_000, 0, 0, 1)])
def test_host_fed_lists_with_empty_batches(sizes):
    # nothing but the wait for its flag stands between an empty batch and the next
    tree, pts = make(), synth.uniform(10, 1 << 16, 2 * sum(sizes))
    for lo in (0, sum(sizes)):
        cut = np.split(pts[lo:lo + sum(sizes)], np.cumsum(sizes)[:-1])
        host = [torch.from_numpy(np.ascontiguousarray(b).view(np.uint8).reshape(-1, 16)).pin_memory()
                for b in cut]
        dst = torch.empty((sum(sizes), 16), dtype=torch.uint8, device="cuda")
        ready = torch.empty(len(sizes), dtype=torch.int32, device="cuda")
        tree.insert_many_host(host, dst, ready, torch.cuda.Stream())
        assert tree.sync() == simlod.OK
    assert tree.progress() == (2 * len(sizes), 2 * len(sizes))
    want = oracle.static_build(oracle.Config.make(**KW), pts)
    assert_snapshots_equal(tree.snapshot(), want)
