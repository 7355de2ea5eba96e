"""Host-buffer calls whose first launch reaches no grid barrier (at most one Laplacian iteration, in a kernel of its own, and
one bilateral pass), with CTAs that have no bilateral tile: the same results as the device call, over and over in one
context whose other calls use the barrier."""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

import paper_2007_12065_gb300 as pl3d  # noqa: E402


@pytest.mark.parametrize("H,W", [(2, 2), (33, 33), (65, 97), (129, 64)])
@pytest.mark.parametrize("lap", [0, 1])
@pytest.mark.parametrize("bil", [0, 2])
def test_host_call_without_a_barrier_in_its_first_launch(H, W, lap, bil):
    f = synth.depth_camera_scene(H, W, seed=H + W, n_boxes=1, noise_sigma=0.004, nan_frac=0.03)
    prm = pl3d.make_params(**dict(f.params, lap_iters=lap, bil_iters=bil))
    nd, n = f.dominant_normals, 2 * (H - 1) * (W - 1)
    ex = pl3d.PlaneExtractor(0)
    # 32-row bilateral tiles: 33 points give four Laplacian tiles (or two) and one bilateral tile
    pl3d.pl3d_set_tuning(ex.ctx, bil_tile_h=32)
    want = {k: v.cpu().numpy() for k, v in ex(torch.from_numpy(f.points).cuda(), prm, nd).items()}
    host = dict(mask=torch.empty(n, dtype=torch.uint8, pin_memory=True),
                normals=torch.empty((n, 3), dtype=torch.float32, pin_memory=True),
                labels=torch.empty(n, dtype=torch.int32, pin_memory=True))
    for _ in range(20):
        for v in host.values():
            v.fill_(7)
        pl3d.pl3d_extract_planes_host(ex.ctx, f.points, H, W, prm, nd, len(nd), host["mask"], host["normals"], host["labels"])
        for k in want:
            np.testing.assert_array_equal(host[k].numpy(), want[k], err_msg=k)
    pl3d.pl3d_sync(ex.ctx)
