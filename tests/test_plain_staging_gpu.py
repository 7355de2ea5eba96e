"""Tiles staged without TMA (odd widths, points at any 4-byte offset, later Laplacian passes): the same points
at an aligned and at a misaligned address give the same bits, and odd widths agree with the same scan inside a TMA-staged
frame away from the cut."""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

import paper_2007_12065_gb300 as pl3d  # noqa: E402


def _run(ex, pts_ptr, H, W, prm, nd):
    n = 2 * (H - 1) * (W - 1)
    o = dict(mask=torch.empty(n, dtype=torch.uint8, device="cuda"), nrm=torch.empty(3 * n, device="cuda"),
             lab=torch.empty(n, dtype=torch.int32, device="cuda"), pts=torch.empty(3 * H * W, device="cuda"))
    pl3d.pl3d_extract_planes_ex(ex.ctx, pts_ptr, H, W, prm, nd, len(nd), o["mask"], o["nrm"], o["lab"], o["pts"], None)
    pl3d.pl3d_sync(ex.ctx)
    return {k: v.cpu().numpy() for k, v in o.items()}


@pytest.mark.parametrize("lap,kernel", [(3, 3), (9, 3), (1, 5)])
@pytest.mark.parametrize("H,W", [(4, 4), (35, 36), (70, 100)])
def test_misaligned_points(H, W, lap, kernel):
    ex = pl3d.PlaneExtractor(0)
    f = synth.depth_camera_scene(H, W, seed=3, n_boxes=1, nan_frac=0.03)
    prm = pl3d.make_params(**dict(f.params, lap_iters=lap, bil_iters=2, lap_kernel=kernel))
    pts = torch.from_numpy(f.points).cuda().reshape(-1)
    want = _run(ex, pts.data_ptr(), H, W, prm, f.dominant_normals)
    room = torch.empty(pts.numel() + 4, device="cuda")
    for off in (1, 2, 3):
        room[off:off + pts.numel()] = pts
        got = _run(ex, room.data_ptr() + 4 * off, H, W, prm, f.dominant_normals)
        for k in want:
            np.testing.assert_array_equal(got[k], want[k], err_msg=f"{k} at offset {off}")


@pytest.mark.parametrize("W", [33, 61, 62, 63, 130])
def test_odd_widths(W):
    # 2 iterations of a 3 x 3 window and 1 of the bilateral reach 4 columns from the cut
    H, Wf = 40, 132
    ex = pl3d.PlaneExtractor(0)
    f = synth.depth_camera_scene(H, Wf, seed=9, n_boxes=1, nan_frac=0.03)
    prm = pl3d.make_params(**dict(f.params, lap_iters=2, bil_iters=1))
    full = _run(ex, torch.from_numpy(f.points).cuda(), H, Wf, prm, f.dominant_normals)
    cut = _run(ex, torch.from_numpy(np.ascontiguousarray(f.points[:, :W])).cuda(), H, W, prm, f.dominant_normals)
    keep = W - 6
    np.testing.assert_array_equal(cut["pts"].reshape(H, W, 3)[:, :keep], full["pts"].reshape(H, Wf, 3)[:, :keep])
    for k, c in (("nrm", 3), ("mask", 1)):
        a, b = cut[k].reshape(H - 1, W - 1, 2, c)[:, :keep], full[k].reshape(H - 1, Wf - 1, 2, c)[:, :keep]
        np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("H,W", [(150, 201), (96, 200)])
def test_many_passes(H, W):
    # the displacement buffers are written and read again by other tiles several times in one launch
    ex = pl3d.PlaneExtractor(0)
    f = synth.depth_camera_scene(H, W, seed=5, n_boxes=1, nan_frac=0.03)
    prm = pl3d.make_params(**dict(f.params, lap_iters=33, bil_iters=1))
    pts = torch.from_numpy(f.points).cuda()
    runs = []
    for fuse in (0, 5, 7):
        pl3d.pl3d_set_tuning(ex.ctx, lap_fuse=fuse)
        runs.append(_run(ex, pts, H, W, prm, f.dominant_normals))
    for other in runs[1:]:
        for k in other:
            np.testing.assert_array_equal(other[k], runs[0][k], err_msg=k)
