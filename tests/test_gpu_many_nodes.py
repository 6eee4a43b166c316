"""Octrees of far more nodes than the GPU has warps (leaves of one to three
points): updates that touch few of them, and updates that split thousands of
leaves at once. Compared with the oracle's closed form byte for byte."""
import numpy as np
import pytest

import oracle
from helpers import assert_snapshots_equal, check_allocator
from paper_2310_03567_gb300 import simlod, synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("form", ["fused", "plain"])
@pytest.mark.parametrize("T,C,G", [(1, 1, 2), (3, 2, 3)])
@pytest.mark.parametrize("cuts", [(60_000, 1, 33, 500, 7), (100, 30_000, 2_000, 28_000)])
def test_updates_of_an_octree_of_many_nodes(form, T, C, G, cuts):
    kw = dict(root_log2=18, leaf_capacity=T, chunk_points=C, grid_log2=G)
    cfg = simlod.default_config(max_batch_points=1 << 16, spill_capacity=1 << 18,
                                backlog_capacity=1 << 20, max_nodes=1 << 20, **kw)
    tree = simlod.Octree(cfg, simlod.make_arena(cfg, 2 << 30), stream=torch.cuda.Stream())
    n = sum(cuts)
    pts = np.concatenate([synth.uniform(31, 1 << 18, n // 2),
                          synth.terrain(32, n - n // 2, extent_m=250.0, row_len=150, root_log2=18)])
    pts = pts[np.random.default_rng(6).permutation(n)]
    batches = [simlod.points_tensor(b) for b in np.split(pts, np.cumsum(cuts)[:-1])]
    if form == "fused":
        tree.insert_many(batches)
    else:
        for b in batches:
            tree.insert(b)
    assert tree.sync() == simlod.OK
    st, got = tree.stats(), tree.snapshot()
    assert st["nodes"] > 20_000
    assert_snapshots_equal(got, oracle.static_build(oracle.Config.make(**kw), pts))
    check_allocator(got, st)
