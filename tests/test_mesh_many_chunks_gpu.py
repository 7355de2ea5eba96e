"""Mesh and segment lists of frames with more chunks than resident CTAs (a CTA's second and third chunk are ranked after
the barrier, its first before it), and two quads per thread at ragged ends."""
import numpy as np
import pytest

import oracle
import synth
from test_mesh_gpu import _check, env  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,W,bands", [(500, 700, 3), (801, 1003, 300), (641, 1281, 2048)])
def test_many_chunks(env, H, W, bands):  # noqa: F811
    """`bands` segments of interleaved triangles: every chunk holds entries of many segments."""
    f = synth.depth_camera_scene(H, W, seed=H + W, n_boxes=2, nan_frac=0.05)
    _, Tmap = oracle.extract_triangles(oracle.widen(f.points))
    valid = np.nonzero(np.asarray(Tmap) >= 0)[0]
    rng = np.random.default_rng(bands)
    band = rng.integers(0, bands, len(valid))
    band[rng.random(len(valid)) < 0.1] = -1
    used, at, which = np.unique(band, return_index=True, return_inverse=True)   # each band's first triangle
    labels = np.full(len(Tmap), -1, np.int32)
    labels[valid] = np.where(band >= 0, valid[at][which], -1)
    dev, _ = _check(env, f.points, labels)
    assert dev["counts"][1] == (used >= 0).sum()
