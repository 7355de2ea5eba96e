"""Tile heights chosen by a frame's size: a single frame under the default tuning, from one quad to several rounds of
tiles, against the same frame at 32-row tiles (every output bit for bit) and, with a 3 x 3 window, against one Laplacian
iteration per pass (the single-iteration kernel)."""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

import paper_2007_12065_gb300 as pl3d  # noqa: E402


@pytest.fixture(scope="module")
def ex():
    return pl3d.PlaneExtractor(0)


def _all(ex, pts, prm, nd, **tuning):
    pl3d.pl3d_set_tuning(ex.ctx, **tuning)
    out = ex(pts, prm, nd, want_points=True, want_groups=True)
    torch.cuda.synchronize()
    pl3d.pl3d_set_tuning(ex.ctx)
    return {k: v.cpu().numpy() for k, v in out.items()}


@pytest.mark.parametrize("H,W,lap,bil,kernel,extra", [
    (2, 2, 2, 1, 3, {}), (3, 40, 5, 3, 3, {}), (9, 33, 2, 2, 3, dict(min_triangles=3)), (17, 257, 6, 4, 3, {}),
    (120, 160, 5, 3, 3, {}), (64, 1024, 3, 2, 3, dict(max_offset=0.02)), (243, 317, 2, 2, 3, dict(min_triangles=25)),
    (500, 500, 2, 2, 5, {}), (130, 131, 1, 2, 7, {}), (721, 1283, 5, 3, 3, {}), (97, 64, 9, 7, 3, {})])
def test_default_heights(ex, H, W, lap, bil, kernel, extra):
    f = synth.depth_camera_scene(H, W, seed=H + W, n_boxes=2, noise_sigma=0.004, nan_frac=0.03)
    prm = pl3d.make_params(**dict(f.params, lap_iters=lap, bil_iters=bil, lap_kernel=kernel, bil_kernel=kernel, **extra))
    pts = torch.from_numpy(f.points).cuda()
    got = _all(ex, pts, prm, f.dominant_normals)
    for tuning in [dict(lap_tile_h=32, bil_tile_h=32)] + ([dict(lap_fuse=1, bil_tile_h=16)] if kernel == 3 and lap <= 8 else []):
        want = _all(ex, pts, prm, f.dominant_normals, **tuning)
        for k in want:
            np.testing.assert_array_equal(got[k], want[k], err_msg=f"{k} {tuning}")
