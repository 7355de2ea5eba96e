"""A second Laplacian pass writes the second half of the displacement scratch with float4 stores: the half
must be 16-byte aligned whatever the first frame of a context was (60 x 100 points once put it at 8 modulo
16). The frame in a new context, against the same frame in a context grown by a larger frame first."""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

import paper_2007_12065_gb300 as pl3d  # noqa: E402


@pytest.mark.parametrize("H,W", [(60, 100), (62, 100), (20, 36), (33, 44)])
def test_second_pass_in_a_new_context(H, W):
    f = synth.depth_camera_scene(H, W, seed=5, n_boxes=2)
    prm = pl3d.make_params(**dict(f.params, lap_iters=9, bil_iters=7))
    pts = torch.from_numpy(f.points).cuda()
    grown = pl3d.PlaneExtractor(0)
    big = synth.depth_camera_scene(120, 160, seed=6, n_boxes=2)
    grown(torch.from_numpy(big.points).cuda(), prm, big.dominant_normals)
    want = grown(pts, prm, f.dominant_normals, want_points=True)
    got = pl3d.PlaneExtractor(0)(pts, prm, f.dominant_normals, want_points=True)
    torch.cuda.synchronize()
    for k in want:
        np.testing.assert_array_equal(got[k].cpu().numpy(), want[k].cpu().numpy(), err_msg=k)
