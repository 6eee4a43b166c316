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
