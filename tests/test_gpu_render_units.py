"""Draw units of the renderer: chunk sizes around the edges of a warp and of a
draw unit's parts, lists whose chunks lie apart (many small batches), a
compacted octree cut into array pieces, and a frame that starts on an 8-byte
boundary. Frames are compared with the CPU renderer bit for bit."""
import numpy as np
import pytest

import oracle
from paper_2310_03567_gb300 import simlod, synth
from test_oracle_render import CAMS, look_at_perspective

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("C,T,batch", [(1, 300, 5_000), (31, 2_000, 777), (33, 2_000, 40_000),
                                       (257, 3_000, 1_500), (1_000, 5_000, 9_999),
                                       (5_000, 9_000, 60_000), (65_536, 20_000, 60_000)])
@pytest.mark.parametrize("compact", [False, True])
def test_frames_for_any_chunk_size(C, T, batch, compact):
    n = 20_000 if C == 1 else 60_000
    pts = np.concatenate([synth.terrain(3, n // 2, extent_m=1000.0, row_len=211, root_log2=20),
                          synth.uniform(4, 1 << 20, n - n // 2)])
    pts = pts[np.random.default_rng(9).permutation(len(pts))]
    cfg = simlod.default_config(root_log2=20, leaf_capacity=T, chunk_points=C, grid_log2=5,
                                max_batch_points=1 << 17, spill_capacity=1 << 20,
                                backlog_capacity=1 << 20, max_nodes=1 << 15)
    tree = simlod.Octree(cfg, simlod.make_arena(cfg, (1 << 30) + (C << 14)),
                         stream=torch.cuda.Stream())
    tree.insert_many([simlod.points_tensor(pts[k:k + batch]) for k in range(0, n, batch)])
    assert tree.sync() == simlod.OK
    ocfg = oracle.Config.make(root_log2=20, leaf_capacity=T, chunk_points=C, grid_log2=5)
    snap = oracle.static_build(ocfg, pts)
    if compact:
        tree.compact()
        if C < 1_000:  # nodes of two chunks and more become arrays
            assert tree.stats()["compact_nodes"] > 0
    W, H = 211, 97  # odd sizes
    for k, (eye, tgt, fov) in enumerate(CAMS):
        m = look_at_perspective(eye, tgt, fov, W / H)
        room = torch.zeros(W * H + 2, dtype=torch.int64, device="cuda")
        fb = room[k & 1:][:W * H].view(H, W)  # 16- and 8-byte aligned in turn
        tree.render(m, fb)
        assert tree.sync() == simlod.OK
        want, drawn, nd = oracle.render(ocfg, snap, m, W, H)
        assert np.array_equal(fb.cpu().numpy().view(np.uint64), want)
        assert int(room[W * H + (k & 1):].abs().sum()) == 0  # nothing past the frame
        st = tree.stats()
        assert st["render_nodes"] == nd
        assert st["render_samples"] == int(np.where(
            snap.nodes["is_inner"] == 1, snap.nodes["n_voxels"], snap.nodes["n_points"])[drawn].sum())


def test_pieces_beyond_the_unit_region_are_drawn_at_once():
    # 1,000 chunks of one octant become an array of 1,000 pieces, and as many
    # points of another octant take the chunks it gave back: 2,000 units in a
    # region that has room for fewer
    C, per = 256, 256_000
    kw = dict(root_log2=20, leaf_capacity=per + 100, chunk_points=C, grid_log2=1)
    cfg = simlod.default_config(max_batch_points=1 << 19, spill_capacity=1 << 16,
                                backlog_capacity=1 << 12, max_nodes=1 << 10, **kw)
    lo = synth.uniform(5, 1 << 19, per)
    hi = synth.uniform(6, 1 << 19, per)
    for f in "xyz":
        hi[f] += 1 << 19
    tree = simlod.Octree(cfg, simlod.make_arena(cfg, 10_570_000), stream=torch.cuda.Stream())
    tree.insert_many([simlod.points_tensor(np.concatenate([lo, hi[:200]]))])
    tree.compact()
    tree.insert_many([simlod.points_tensor(hi[200:])])
    assert tree.sync() == simlod.OK
    st = tree.stats()
    assert st["compact_nodes"] == 1 and st["compact_chunks"] == per // C
    assert st["data_bytes"] // (20 * C + 256) < 2 * per // C  # chunks in the data region
    ocfg = oracle.Config.make(**kw)
    snap = oracle.static_build(ocfg, np.concatenate([lo, hi]))
    eye, tgt, fov = CAMS[0]
    W, H = 211, 97
    m = look_at_perspective(eye, tgt, fov, W / H)
    fb = torch.empty((H, W), dtype=torch.int64, device="cuda")
    tree.render(m, fb)
    assert tree.sync() == simlod.OK
    want, drawn, nd = oracle.render(ocfg, snap, m, W, H)
    assert np.array_equal(fb.cpu().numpy().view(np.uint64), want)
    assert tree.stats()["render_nodes"] == nd


def test_captured_frames_and_compactions():
    # a captured render draws the octree as it is at each replay, a captured
    # compaction compacts it
    kw = dict(root_log2=20, leaf_capacity=700, chunk_points=50, grid_log2=5)
    cfg = simlod.default_config(max_batch_points=1 << 16, spill_capacity=1 << 18,
                                backlog_capacity=1 << 18, max_nodes=1 << 14, **kw)
    pts = synth.uniform(7, 1 << 20, 40_000)
    tree = simlod.Octree(cfg, simlod.make_arena(cfg, 256 << 20))
    eye, tgt, fov = CAMS[0]
    m = look_at_perspective(eye, tgt, fov, 2.0)
    fb, direct = (torch.empty((128, 256), dtype=torch.int64, device="cuda") for _ in range(2))
    tree.render(m, direct)
    tree.compact()
    torch.cuda.synchronize()
    frame, pack = torch.cuda.CUDAGraph(), torch.cuda.CUDAGraph()
    with torch.cuda.graph(frame):
        tree.render(m, fb)
    with torch.cuda.graph(pack):
        tree.compact()
    for lo in (0, 20_000):
        tree.insert(simlod.points_tensor(pts[lo:lo + 20_000]))
        pack.replay()
        frame.replay()
        tree.render(m, direct)
        assert tree.sync() == simlod.OK
        assert tree.stats()["compact_nodes"] > 0
        assert torch.equal(fb, direct) and bool((fb != -1).any())
    ocfg = oracle.Config.make(**kw)
    want, _, _ = oracle.render(ocfg, oracle.static_build(ocfg, pts), m, 256, 128)
    assert np.array_equal(fb.cpu().numpy().view(np.uint64), want)
