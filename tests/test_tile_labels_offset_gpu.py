"""Segments inside a tile with the plane-offset test on, against the oracle's region growing of the same groups with the same
test on FP64 centroids: steps between plateaus that break the diagonal, the right and the upper link of a quad, on
the scans of test_tile_labels_gpu.py. The offsets stay clear of the limit (1e-4 of 7.5e-3, where FP32 centroids of these
coordinates are off by 1e-5 at most), so the labels are equal."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

import paper_2007_12065_gb300 as pl3d  # noqa: E402
from test_tile_labels_gpu import _walls  # noqa: E402

LIMIT = 7.5e-3


@pytest.mark.parametrize("bil_tile_h", [8, 16, 24, 32])
@pytest.mark.parametrize("kind", ["open", "serpentine", "comb_down", "comb_up", "spiral", "holes"])
def test_tile_segments_with_offsets(kind, bil_tile_h):
    H, W = 71, 103
    rng = np.random.default_rng(12)
    u, v = np.mgrid[0:H, 0:W]
    # plateaus 3 x 4 points: a centroid moves by a third of a step, 4, 11 or 15 mm
    level = np.array([0.0, 0.0, 0.012, 0.045])[rng.integers(0, 4, (H // 3 + 1, W // 4 + 1))]
    z = level[u // 3, v // 4] + 1e-4 * rng.standard_normal((H, W))
    pts = np.stack([0.2 * v, 0.2 * u, z], -1).astype(np.float32)
    pts[_walls(kind, H, W)] = np.nan
    nd = np.array([[0, 0, 1], [0, 0, -1]], np.float32)
    prm = dict(lap_iters=0, bil_iters=0, max_edge=0.0, min_dot=0.9, max_offset=LIMIT)
    n = 2 * (H - 1) * (W - 1)
    dev = dict(device="cuda")
    mask, grp = torch.empty(n, dtype=torch.uint8, **dev), torch.empty(n, dtype=torch.uint8, **dev)
    nrm, lab = torch.empty(3 * n, dtype=torch.float32, **dev), torch.empty(n, dtype=torch.int32, **dev)
    ctx = pl3d.pl3d_create(0)
    try:
        pl3d.pl3d_set_tuning(ctx, bil_tile_h=bil_tile_h)
        pl3d.pl3d_extract_planes_ex(ctx, torch.from_numpy(pts).cuda(), H, W, pl3d.make_params(**prm), nd, len(nd), mask, nrm,
                                    lab, None, grp)
        pl3d.pl3d_sync(ctx)
    finally:
        pl3d.pl3d_destroy(ctx)
    g = grp.cpu().numpy()
    c = oracle.extract_planes(pts, oracle.OracleParams(**prm), nd, sensitivity=False)["centroids"].reshape(H - 1, W - 1, 2, 3)
    gq, cz = g.reshape(H - 1, W - 1, 2), c[..., 2]
    pairs = [(gq[..., 0], gq[..., 1], cz[..., 0] - cz[..., 1]),                              # the quad's diagonal
             (gq[:, :-1, 0], gq[:, 1:, 1], cz[:, :-1, 0] - cz[:, 1:, 1]),                    # first(v), second(v + 1)
             (gq[1:, :, 0], gq[:-1, :, 1], cz[1:, :, 0] - cz[:-1, :, 1])]                    # first(r), second(r - 1)
    for ga, gb, d in pairs:
        d = np.abs(d[(ga == gb) & (ga != pl3d.PL3D_NO_GROUP)])
        assert (d > LIMIT).sum() > 20 and (d <= LIMIT).sum() > 20
        assert np.abs(d - LIMIT).min() > 1e-4
    want = oracle.label(g, H, W, C=c.reshape(-1, 3), nd_unit=nd.astype(np.float64), max_offset=LIMIT)
    assert not np.array_equal(want, oracle.label(g, H, W))
    np.testing.assert_array_equal(lab.cpu().numpy(), want)
