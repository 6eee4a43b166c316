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


def alone(what):
    """Counters after the failing launch with nothing behind it."""
    tree, batches, status = failing(what)
    tree.insert_many(batches)
    assert tree.sync() == status
    return tree.stats()


@pytest.mark.parametrize("what", ["arena", "nodes"])
@pytest.mark.parametrize("behind", ["one", "many", "budget", "hostfed", "plan", "rejected"])
def test_update_behind_a_failed_update(what, behind):
    want = alone(what)
    tree, batches, status = failing(what)
    ptrs = [b.data_ptr() for b in batches]
    counts = [len(b) for b in batches]
    plan = tree.plan(ptrs, counts, merge_points=20_000) if behind == "plan" else None
    out = PTS[:10].copy()
    out["z"][4] = -1  # outside the root cube
    bad = simlod.points_tensor(out)
    host = [b.cpu().pin_memory() for b in batches[:3]]
    dst = torch.empty((15_000, 16), dtype=torch.uint8, device="cuda")
    ready = torch.zeros(3, dtype=torch.int32, device="cuda")
    copies = torch.cuda.Stream()
    torch.cuda.synchronize()
    tree.insert_many(batches)
    for _ in range(2):
        if behind == "one":
            tree.insert_many(batches[:1])
        elif behind == "many":
            tree.insert_many(batches)
        elif behind == "budget":
            assert tree.insert_many_ptrs(ptrs, counts, budget_ns=10 ** 9) == simlod.OK
        elif behind == "hostfed":
            tree.insert_many_host(host, dst, ready, copies)
        elif behind == "plan":
            assert plan.run() == simlod.OK
        else:
            tree.insert_many([bad])
    assert tree.sync() == status
    got = tree.stats()
    for k in ("batches", "points", "rejected_batches", "splits", "voxels", "last_points"):
        assert got[k] == want[k], k
    works_after_reset(tree)
    if plan:
        plan.close()


def test_plain_update_behind_a_failed_update():
    tree, batches, status = failing("nodes")
    want = alone("nodes")
    tree.insert_many(batches)
    assert tree.insert(batches[0], check=False) == status
    assert tree.insert(batches[0], check=False) == simlod.ERR_POISONED
    assert tree.stats()["batches"] == want["batches"]
    works_after_reset(tree)


@pytest.mark.parametrize("what", ["arena", "nodes"])
@pytest.mark.parametrize("clear", [True, False])
def test_frame_behind_a_failed_update(what, clear):
    # the frame is cleared as asked, and no node is drawn
    tree, batches, status = failing(what)
    side = float(1 << 16)
    cam = simlod.view_proj([side * 0.1] * 3, [side / 2] * 3, 90.0, 2.0)
    frame = torch.full((128, 256), 77, dtype=torch.int64, device="cuda")
    tree.insert_many(batches)
    tree.render(cam, frame, clear=clear)
    assert tree.sync() == status
    assert bool((frame == (-1 if clear else 77)).all())
    st = tree.stats()
    assert st["render_nodes"] == st["render_samples"] == 0
    works_after_reset(tree)
    tree.render(cam, frame)
    assert tree.sync() == simlod.OK and bool((frame != -1).any())


@pytest.mark.parametrize("what", ["arena", "nodes"])
@pytest.mark.parametrize("synced", [True, False])
def test_restore_behind_a_failed_update(what, synced):
    # the failed update's counts and claims are gone with its octree, whether its
    # status has been read or not
    tree, batches, status = failing(what)
    tree.insert_many(batches[:1])
    snap = tree.snapshot()
    tree.reset()
    tree.insert_many(batches)
    if synced:
        assert tree.sync() == status
    tree.restore(snap)
    tree.insert_many(batches[1:2])
    assert tree.sync() == simlod.OK
    want = oracle.static_build(oracle.Config.make(**KW), PTS[:10_000])
    assert_snapshots_equal(tree.snapshot(), want)
