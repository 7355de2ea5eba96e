"""The flatten phase of a batch (blocks of 1024 labels per warp, eight 16-byte loads per lane): frames around the block
edges, labels buffers at every 4-byte offset, segment sizes counted or not, against the same frames run alone."""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

import paper_2007_12065_gb300 as pl3d  # noqa: E402

# 2 (H-1)(W-1) labels: 2, 1020, 1022, 1024, 1026, 2046, 2050, several blocks
SIZES = [(2, 2), (11, 52), (8, 74), (5, 129), (20, 28), (34, 32), (6, 206), (97, 131)]


@pytest.mark.parametrize("tri_min", [0, 4])
@pytest.mark.parametrize("off", [0, 1, 2, 3])
def test_batch_labels(off, tri_min):
    ex = pl3d.PlaneExtractor(0)
    batch, rooms, want = pl3d.Batch(), [], []
    for H, W in SIZES:
        f = synth.depth_camera_scene(H, W, seed=1000 * H + W, n_boxes=2, noise_sigma=0.004, nan_frac=0.03)
        prm = pl3d.make_params(**dict(f.params, lap_iters=1, bil_iters=1, max_edge=0.0, min_dot=0.8,
                                      min_triangles=tri_min))
        n = 2 * (H - 1) * (W - 1)
        pts = torch.from_numpy(f.points).cuda()
        want.append(ex(pts, prm, f.dominant_normals)["labels"].cpu().numpy())
        room = torch.full((n + 8,), -7, dtype=torch.int32, device="cuda")
        rooms.append(room)
        batch.add(pts, H, W, prm, f.dominant_normals, torch.empty(n, dtype=torch.uint8, device="cuda"),
                  torch.empty(3 * n, device="cuda"), room[off:off + n])
    pl3d.pl3d_extract_planes_batched(ex.ctx, batch)
    pl3d.pl3d_sync(ex.ctx)
    for room, w in zip(rooms, want):
        got = room.cpu().numpy()
        np.testing.assert_array_equal(got[off:off + len(w)], w)
        assert (got[:off] == -7).all() and (got[off + len(w):] == -7).all()
