"""The default launch shape of a batch does not depend on whether two CTAs per SM are asked for or left open (both mean as
many as fit): a batch large enough for one Laplacian iteration per pass runs those passes either way. The autotuner times
that shape beside its own candidates."""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

import paper_2007_12065_gb300 as pl3d  # noqa: E402

KEYS = ("mask", "normals", "labels")


def _batch(frames, params):
    """A batch over (host points, dominant normals) with outputs of its own per frame."""
    b, outs = pl3d.Batch(), []
    for p, nd in frames:
        H, W = p.shape[:2]
        n = 2 * (H - 1) * (W - 1)
        o = dict(mask=torch.empty(n, dtype=torch.uint8, device="cuda"),
                 normals=torch.empty((n, 3), dtype=torch.float32, device="cuda"),
                 labels=torch.empty(n, dtype=torch.int32, device="cuda"))
        b.add(p, H, W, pl3d.make_params(**params), nd, o["mask"], o["normals"], o["labels"])
        outs.append(o)
    return b, outs


def test_two_ctas_per_sm_is_the_default():
    f = synth.depth_camera_scene(480, 640, seed=3, n_boxes=4, noise_sigma=0.005, nan_frac=0.03)
    pts = torch.from_numpy(f.points).cuda()
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    frames = [(pts, f.dominant_normals)] * int(60 * sms / 152)   # 18 million points on 152 SMs
    ctx = pl3d.pl3d_create(0)
    try:
        launches, got = {}, {}
        for c in (0, 2, 1):
            pl3d.pl3d_set_tuning(ctx, ctas_per_sm=c)
            b, outs = _batch(frames, dict(f.params, lap_iters=3, bil_iters=1))
            n0 = pl3d.pl3d_launch_count(ctx)
            pl3d.pl3d_extract_planes_batched(ctx, b)
            pl3d.pl3d_sync(ctx)
            launches[c] = pl3d.pl3d_launch_count(ctx) - n0
            got[c] = {k: outs[-1][k].cpu().numpy() for k in KEYS}
        # three single-iteration passes and the batch kernel, or with one CTA per SM the batch kernel alone
        assert launches == {0: 4, 2: 4, 1: 1}
        for c in (2, 1):
            for k in KEYS:
                np.testing.assert_array_equal(got[c][k], got[0][k], err_msg=f"{k} {c}")
    finally:
        pl3d.pl3d_destroy(ctx)


@pytest.mark.parametrize("kernel,lap,candidates", [
    # 3 x 3: the untuned shape (all three iterations in 64-row tiles), then 3, 1 and 2 iterations per pass at one and two
    # CTAs per SM; 5 x 5: the untuned shape is the fused one at two CTAs per SM; then 12 heights less the timed one
    (3, 3, 1 + 3 * 2 + 11), (5, 2, 2 * 2 + 11)])
def test_autotuner_times_the_untuned_shape(kernel, lap, candidates):
    f = synth.depth_camera_scene(120, 160, seed=4, n_boxes=2, noise_sigma=0.005, nan_frac=0.03)
    pts = torch.from_numpy(f.points).cuda()
    ctx = pl3d.pl3d_create(0)
    try:
        b, outs = _batch([(pts, f.dominant_normals)] * 2, dict(f.params, lap_iters=lap, bil_iters=1, lap_kernel=kernel))
        n0 = pl3d.pl3d_batch_stats(ctx)["graph_launches"]
        pl3d.pl3d_autotune_batched(ctx, b, reps=1)
        # every candidate untimed and timed once, and the choice once more
        assert pl3d.pl3d_batch_stats(ctx)["graph_launches"] - n0 == 2 * candidates + 1
        tuned = {k: outs[0][k].cpu().numpy() for k in KEYS}
        pl3d.pl3d_set_tuning(ctx, None)
        pl3d.pl3d_extract_planes_batched(ctx, b)
        pl3d.pl3d_sync(ctx)
        for k in KEYS:
            np.testing.assert_array_equal(tuned[k], outs[0][k].cpu().numpy(), err_msg=k)
    finally:
        pl3d.pl3d_destroy(ctx)
