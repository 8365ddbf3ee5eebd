"""The scatter kernels' clipping and pixel arithmetic at their edges (GPU only),
bit for bit against the oracle: cameras inside, above, under and beside the
sampled ground, columns that cross the camera's plane and the image's borders,
flat ground (a column of one point), the fewest and the most points, images of
one pixel, one row and one column."""

import numpy as np
import pytest

import synth
from oracle import scatter as oscatter
from test_gpu_scatter import _check, _run, hf  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nu,nv,nz", [(200, 150, 2), (64, 64, 33), (97, 61, 300), (16, 16, 4096)])
@pytest.mark.parametrize("flat", (False, True))
def test_columns_across_the_image(hf, nu, nv, nz, flat):
    W, H = 120, 90
    cells, _ = synth.make_grid(W, H, seed=nz, slab_frac=0.4, n_walls=9)
    if flat:
        cells = cells & np.uint32(0xFF000000)
    cams = synth.camera_array([
        synth.pose_to_camera(60.0, 45.0, 30.0, 20.0, 0.0, 90, 64, 48),    # inside the ground
        synth.pose_to_camera(60.5, 45.5, 125.0, 110.0, -89.0, 60, 33, 65),
        synth.pose_to_camera(5.0, 5.0, 260.0, 45.0, -20.0, 120, 57, 1),
        synth.pose_to_camera(100.0, 80.0, 90.0, 250.0, 25.0, 2, 1, 57),
        synth.pose_to_camera(30.0, 60.0, 0.0, 180.0, 5.0, 60, 1, 1),
        synth.pose_to_camera(64.0, 32.0, 64.0, 0.0, -45.0, 90, 128, 96),
    ])
    fps = synth.footprints(cams)
    ctx = hf.hf_create(cells)
    try:
        raw = _run(hf, ctx, cams, fps, nu, nv, nz, 700.0, raw=True)
        got = _run(hf, ctx, cams, fps, nu, nv, nz, 700.0)
        for i, cam in enumerate(cams):
            want = oscatter.render(cells, cam, nu, nv, nz, *[float(v) for v in fps[i]], 700.0)
            assert np.array_equal(raw[i]["hit_cell"], want["packed"]), "screen %d" % i
            _check(got[i], want, "camera %d" % i)
    finally:
        hf.hf_destroy(ctx)
