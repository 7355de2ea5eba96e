"""The flatten phase's blocks (256 labels per warp, 16-byte accesses from the buffer's own alignment):
frames around the block edges and labels buffers at every 4-byte offset, against the oracle's region
growing of the groups that the same call wrote (whole numbers, equal), the offset buffer's neighbours
untouched; and the host-buffer call's second copy of the labels."""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

import paper_2007_12065_gb300 as pl3d  # noqa: E402


@pytest.fixture(scope="module")
def ctx():
    c = pl3d.pl3d_create(0)
    yield c
    pl3d.pl3d_destroy(c)


def _scene(H, W):
    return synth.depth_camera_scene(H, W, seed=1000 * H + W, n_boxes=2, noise_sigma=0.004, nan_frac=0.03)


# 2 (H-1)(W-1) labels: 2, 254, 256, 258, 260, 510, 514, a few blocks, several blocks per warp
SIZES = [(2, 2), (2, 128), (2, 129), (4, 44), (2, 131), (6, 52), (2, 258), (41, 67), (333, 389), (700, 903)]


@pytest.mark.parametrize("tri_min", [0, 4])
@pytest.mark.parametrize("H,W", SIZES)
def test_labels_at_every_offset(ctx, H, W, tri_min):
    f = _scene(H, W)
    nd = f.dominant_normals
    prm = pl3d.make_params(**dict(f.params, lap_iters=1, bil_iters=1, max_edge=0.0, min_dot=0.8, min_triangles=tri_min))
    n = 2 * (H - 1) * (W - 1)
    pts = torch.from_numpy(f.points).cuda()
    mask = torch.empty(n, dtype=torch.uint8, device="cuda")
    nrm = torch.empty(3 * n, dtype=torch.float32, device="cuda")
    grp = torch.empty(n, dtype=torch.uint8, device="cuda")
    for off in range(4):
        room = torch.full((n + 8,), -7, dtype=torch.int32, device="cuda")
        pl3d.pl3d_extract_planes_ex(ctx, pts, H, W, prm, nd, len(nd), mask, nrm, room.data_ptr() + 4 * off, None, grp)
        pl3d.pl3d_sync(ctx)
        want = oracle.label(grp.cpu().numpy(), H, W, tri_min=tri_min)
        got = room.cpu().numpy()
        np.testing.assert_array_equal(got[off:off + n], want)
        assert (got[:off] == -7).all() and (got[off + n:] == -7).all()


@pytest.mark.parametrize("off", [0, 1, 2])
def test_host_labels_copy(ctx, off):
    H, W = 97, 131
    f = _scene(H, W)
    prm = pl3d.make_params(**dict(f.params, lap_iters=1, bil_iters=1))
    n = 2 * (H - 1) * (W - 1)
    want = pl3d.PlaneExtractor(0)(torch.from_numpy(f.points).cuda(), prm, f.dominant_normals)["labels"].cpu().numpy()
    pts = torch.from_numpy(f.points).pin_memory()
    mask = torch.empty(n, dtype=torch.uint8, pin_memory=True)
    nrm = torch.empty(3 * n, dtype=torch.float32, pin_memory=True)
    room = torch.full((n + 8,), -7, dtype=torch.int32, pin_memory=True)
    pl3d.pl3d_extract_planes_host(ctx, pts, H, W, prm, f.dominant_normals, len(f.dominant_normals), mask, nrm,
                                  room[off:off + n])
    got = room.numpy()
    np.testing.assert_array_equal(got[off:off + n], want)
    assert (got[:off] == -7).all() and (got[off + n:] == -7).all()
