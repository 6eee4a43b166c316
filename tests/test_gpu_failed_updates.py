"""What is enqueued behind an asynchronous update that fails, before the host
has learned of it: nothing touches the octree, and the next sync reports the
update's own error."""
import pytest

import oracle
from helpers import assert_snapshots_equal
from paper_2310_03567_gb300 import simlod, synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

KW = dict(root_log2=16, leaf_capacity=200, chunk_points=16, grid_log2=7)
PTS = synth.uniform(37, 1 << 16, 200_000)


def failing(what):
    """An octree, and batches of which the later ones do not fit it."""
    cfg = simlod.default_config(max_batch_points=1 << 20, spill_capacity=1 << 20,
                                backlog_capacity=1 << 21,
                                max_nodes=1_000 if what == "nodes" else 1 << 16, **KW)
    data = {"arena": 24 << 20, "nodes": 256 << 20}[what]
    tree = simlod.Octree(cfg, simlod.make_arena(cfg, data), stream=torch.cuda.Stream())
    status = {"arena": simlod.ERR_ARENA_FULL, "nodes": simlod.ERR_NODES_FULL}[what]
    return tree, [simlod.points_tensor(PTS[k:k + 5_000]) for k in range(0, len(PTS), 5_000)], status


def works_after_reset(tree):
    tree.reset()
    tree.insert_many([simlod.points_tensor(PTS[:300])])
    assert tree.sync() == simlod.OK
    assert_snapshots_equal(tree.snapshot(), oracle.static_build(oracle.Config.make(**KW), PTS[:300]))


@pytest.mark.parametrize("what", ["arena", "nodes"])
def test_compaction_behind_a_failed_update(what):
    tree, batches, status = failing(what)
    tree.insert_many(batches)
    tree.compact()
    assert tree.sync() == status
    st = tree.stats()
    assert 0 < st["batches"] < len(batches)
    assert st["compacted_total"] == st["compact_nodes"] == 0
    works_after_reset(tree)
