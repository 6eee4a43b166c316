"""The part of an arena in front of its data region never grows beyond what the
library used to place there, so that an arena of a size asked for then holds
what it held."""
import math
import random

import pytest

from paper_2310_03567_gb300 import simlod


def up(v, a=256):
    return (v + a - 1) // a * a


def former_arena_bytes(kw, data):
    """simlod_arena_bytes of the layout with two lists of movers and the records of
    re-inserted points."""
    n, b, s = kw["max_nodes"], kw["max_batch_points"], kw["spill_capacity"]
    bl = kw["backlog_capacity"]
    slots = 1 << max(0, (2 * bl - 1).bit_length())
    o = 0
    for r in (1408, 64, 24 * 16_384, 4 * n, 4 * n, 4 * n, 4 * n, 64 * n, 8 * (n // 8 + 1), 4 * s,
              4 * b, 8 * (b + s), 8 * (b + s), 16 * s, 4 * s, 4 * n, 4 * n, 16 * slots, 4 * bl,
              16 * b):
        o = up(o) + r
    chunks = data // up(16 + 20 * kw["chunk_points"]) + 1
    o = up(o) + 3 * up(4 * chunks) + up(16 * chunks) + 256
    return up(o + data) + 256


def test_the_fixed_part_stays_within_its_former_size():
    rng = random.Random(4)

    def log(lo, hi):
        return int(math.exp(rng.uniform(math.log(lo), math.log(hi))))

    for k in range(3_000):
        kw = dict(root_log2=20, leaf_capacity=log(1, 200_000), chunk_points=log(4, 65_536),
                  grid_log2=rng.randint(1, 7), max_batch_points=log(1, 1 << 30),
                  spill_capacity=log(1, 1 << 30) if rng.random() < 0.9 else 0,
                  backlog_capacity=log(1, 1 << 30), max_nodes=log(9, 1 << 27))
        data = log(1, 1 << 36)
        assert simlod.arena_bytes(simlod.default_config(**kw), data) <= \
            former_arena_bytes(kw, data), kw


@pytest.mark.gpu
@pytest.mark.parametrize("B,S,backlog", [(6_000, 0, 1 << 20), (1_500, 4_500, 1 << 18),
                                         (1_500, 5_000, 1 << 18), (700, 20_000, 40_000)])
@pytest.mark.parametrize("T,C,G", [(1, 4, 2), (40, 7, 4), (5_000, 100, 6)])
def test_arenas_of_the_former_size(B, S, backlog, T, C, G):
    # backlogs that dwarf the batches leave no room, or not enough, for the list of
    # the new voxels' nodes and for histograms of more than a level or two
    import numpy as np
    import torch

    import oracle
    from helpers import assert_snapshots_equal, check_allocator
    from paper_2310_03567_gb300 import synth

    kw = dict(root_log2=14, leaf_capacity=T, chunk_points=C, grid_log2=G, max_batch_points=B,
              spill_capacity=S, backlog_capacity=backlog, max_nodes=1 << 17)
    data = 192 << 20
    n = 15_000 if S > 15_000 else 4_500  # (an update re-inserts at most all of them)
    pts = np.concatenate([synth.uniform(41, 1 << 14, n // 2),
                          synth.uniform(42, 1 << 9, n - n // 2)])
    pts = pts[np.random.default_rng(1).permutation(n)]
    size = n if S == 0 else B
    arena = torch.empty(former_arena_bytes(kw, data), dtype=torch.uint8, device="cuda")
    tree = simlod.Octree(simlod.default_config(**kw), arena, stream=torch.cuda.Stream())
    batches = [simlod.points_tensor(pts[k:k + size]) for k in range(0, n, size)]
    okw = {k: kw[k] for k in ("root_log2", "leaf_capacity", "chunk_points", "grid_log2")}
    want = oracle.static_build(oracle.Config.make(**okw), pts)
    for form in ("fused", "plain"):
        tree.reset()
        if form == "fused":
            tree.insert_many(batches)
        else:
            for b in batches:
                tree.insert(b)
        assert tree.sync() == simlod.OK
        got, st = tree.snapshot(), tree.stats()
        assert st["data_bytes"] >= data
        assert_snapshots_equal(got, want)
        check_allocator(got, st)
