"""Where a voxel traversal starts (GPU only), against the oracle: step limits
around the number of levels, cameras inside a solid, on voxel planes, at the
box's edge and outside it, extents that are no power of two, few and many levels."""

import numpy as np
import pytest

import oracle
import synth
from oracle import voxel as ovox
from test_gpu_voxel import _compare, _levels_for, _rand_grid, _render, hf  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("v,levels", [((4, 8, 2), 0), ((3, 5, 7), 0), ((1, 1, 1), 0), ((6, 4, 3), 2),
                                      ((4, 4, 4), 12), ((64, 64, 256), 0)])
def test_start_level_and_step_limit(hf, v, levels):
    rng = np.random.default_rng(sum(v))
    W, H = 75, 66
    cells = _rand_grid(rng, W, H)
    spots = [(33.3, 20.2, 150.0), (33.3, 20.2, 2.0), (36.0, 24.0, 84.0), (0.0, 0.0, 0.0),
             (74.996, 65.99, 254.0), (12.0, 40.0, 256.0), (40.5, 8.25, 700.0)]
    cams = [synth.pose_to_camera(*p, 41.0 + 50 * i, -20.0, 70, 17, 9) for i, p in enumerate(spots)]
    ctx = hf.hf_create(cells)
    try:
        hf.hf_voxel_build(ctx, *v, levels)
        L = levels or _levels_for(-(-W // v[0]), -(-H // v[1]), -(-256 // v[2]))
        g = ovox.Grid(cells, *v, L)
        cams = synth.camera_array(cams)
        for outer in [1, 2, L - 1, L, L + 1, L + 4, 300]:
            if outer < 1:
                continue
            got = _render(hf, ctx, cams, hf.make_voxel_opts(outer=outer, inner=3, far_dist=400.0))
            for i, cam in enumerate(cams):
                want = ovox.trace(g, cam["o"], oracle.ray_dirs(cam), far=400.0, outer=outer, inner=3)
                _compare(got[i], want, "v %s outer %d cam %d" % (v, outer, i))
    finally:
        hf.hf_destroy(ctx)
