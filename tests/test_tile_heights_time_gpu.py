"""Tile heights of a single frame are chosen for both phases together: a Laplacian height whose tiles outnumber the SMs puts
two CTAs on some of them, and a bilateral phase with fewer tiles than SMs then takes as long as two tiles
on one SM. The chosen heights are not slower than 32 rows for both, in the same process (outputs at any height are compared in
test_tile_heights_gpu.py)."""
import pytest

import synth

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

import paper_2007_12065_gb300 as pl3d  # noqa: E402


def _us(fn, n=30):
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    best = float("inf")
    for _ in range(6):
        e0.record()
        for _ in range(n):
            fn()
        e1.record()
        torch.cuda.synchronize()
        best = min(best, e0.elapsed_time(e1) / n * 1e3)
    return best


# 57 or 60 columns of tiles: two rows of bilateral tiles fit 152 SMs, three or four rows of Laplacian tiles do not
@pytest.mark.parametrize("H,W", [(48, 1800), (49, 1800), (43, 1916)])
def test_chosen_heights_are_not_slower_than_32_rows(H, W):
    if torch.cuda.get_device_properties(0).multi_processor_count < 120:
        pytest.skip("shapes chosen for 120 SMs or more")
    f = synth.depth_camera_scene(H, W, seed=1, n_boxes=2, noise_sigma=0.004, nan_frac=0.03)
    pts = torch.from_numpy(f.points).cuda()
    prm = pl3d.make_params(**dict(f.params, lap_iters=8, bil_iters=5))
    nd, n = f.dominant_normals, 2 * (H - 1) * (W - 1)
    m, l = torch.empty(n, dtype=torch.uint8, device="cuda"), torch.empty(n, dtype=torch.int32, device="cuda")
    v = torch.empty((n, 3), device="cuda")
    ctx = pl3d.pl3d_create(0)
    try:
        def time_at(**tuning):
            pl3d.pl3d_set_tuning(ctx, **tuning)
            return _us(lambda: pl3d.pl3d_extract_planes(ctx, pts, H, W, prm, nd, len(nd), m, v, l))

        time_at()
        chosen, fixed = time_at(), time_at(lap_tile_h=32, bil_tile_h=32)
        pl3d.pl3d_sync(ctx)
    finally:
        pl3d.pl3d_destroy(ctx)
    print(f"{H}x{W}: {chosen:.1f} us chosen, {fixed:.1f} us at 32 rows")
    assert chosen <= 1.05 * fixed
