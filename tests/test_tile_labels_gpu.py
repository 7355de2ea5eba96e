"""Segments inside a tile, in rounds over all links at once: scans cut by missing points into shapes
that need several rounds (a serpentine through every tile, a spiral, combs whose teeth meet at either end, random
holes), at every tile height, against the oracle's region growing of the groups that the same call
wrote (whole numbers, equal)."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

import paper_2007_12065_gb300 as pl3d  # noqa: E402


@pytest.fixture(scope="module")
def ctx():
    c = pl3d.pl3d_create(0)
    yield c
    pl3d.pl3d_destroy(c)


def _walls(kind, H, W):
    """Missing points [H, W]."""
    m = np.zeros((H, W), bool)
    u, v = np.mgrid[0:H, 0:W]
    if kind == "serpentine":        # corridors two quads wide, joined left and right in turn
        m = (u % 3 == 2) & np.where((u // 3) % 2 == 0, v < W - 3, v > 2)
    elif kind == "comb_down":       # teeth joined only at the bottom
        m = (v % 3 == 2) & (u < H - 3)
    elif kind == "comb_up":
        m = (v % 3 == 2) & (u > 2)
    elif kind == "spiral":
        r0, r1, c0, c1 = 0, H - 1, 0, W - 1
        while r1 - r0 > 8 and c1 - c0 > 8:
            m[r0 + 3, c0:c1 - 2] = True
            m[r0 + 3:r1 - 2, c1 - 3] = True
            m[r1 - 3, c0 + 3:c1 - 2] = True
            m[r0 + 6:r1 - 2, c0 + 3] = True
            r0, r1, c0, c1 = r0 + 3, r1 - 3, c0 + 3, c1 - 3
    elif kind == "holes":
        m = np.random.default_rng(H * 1000 + W).random((H, W)) < 0.22
    return m


@pytest.mark.parametrize("max_offset", [0.0, 0.01])
@pytest.mark.parametrize("bil_tile_h", [8, 16, 24, 32])
@pytest.mark.parametrize("kind", ["serpentine", "comb_down", "comb_up", "spiral", "holes"])
def test_tile_segments(ctx, kind, bil_tile_h, max_offset):
    H, W = 71, 103
    rng = np.random.default_rng(11)
    u, v = np.mgrid[0:H, 0:W].astype(np.float32)
    z = (0.3 * np.sin(u / 9.0) * np.cos(v / 7.0) if kind == "holes" else 0.0 * u) + 1e-4 * rng.standard_normal((H, W))
    pts = np.stack([0.05 * v, 0.05 * u, z], -1).astype(np.float32)
    pts[_walls(kind, H, W)] = np.nan
    nd = np.array([[0, 0, 1], [0, 0.5, 1], [0.5, 0, 1], [0, 0, -1], [0, -0.5, -1]], np.float32)
    prm = pl3d.make_params(lap_iters=0, bil_iters=0, max_edge=0.0, min_dot=0.9, max_offset=max_offset)
    n = 2 * (H - 1) * (W - 1)
    dev = dict(device="cuda")
    mask, grp = torch.empty(n, dtype=torch.uint8, **dev), torch.empty(n, dtype=torch.uint8, **dev)
    nrm, lab = torch.empty(3 * n, dtype=torch.float32, **dev), torch.empty(n, dtype=torch.int32, **dev)
    pl3d.pl3d_set_tuning(ctx, bil_tile_h=bil_tile_h)
    pl3d.pl3d_extract_planes_ex(ctx, torch.from_numpy(pts).cuda(), H, W, prm, nd, len(nd), mask, nrm, lab, None, grp)
    pl3d.pl3d_sync(ctx)
    pl3d.pl3d_set_tuning(ctx)
    g = grp.cpu().numpy()
    assert (g != pl3d.PL3D_NO_GROUP).sum() > n // 8
    if max_offset > 0:
        # the offset test compares centroids in FP32: the same segments at every tile height
        one = torch.empty_like(lab)
        pl3d.pl3d_set_tuning(ctx, bil_tile_h=8 if bil_tile_h != 8 else 32)
        pl3d.pl3d_extract_planes(ctx, torch.from_numpy(pts).cuda(), H, W, prm, nd, len(nd), mask, nrm, one)
        pl3d.pl3d_sync(ctx)
        pl3d.pl3d_set_tuning(ctx)
        np.testing.assert_array_equal(lab.cpu().numpy(), one.cpu().numpy())
    else:
        np.testing.assert_array_equal(lab.cpu().numpy(), oracle.label(g, H, W))
