"""Cameras just above the occupancy box (GPU only), against the oracle: where an
extent does not divide 256 the last voxels of coarse levels reach past the box,
so a camera outside it can lie in a voxel of every level above the lowest.  Its
rays start where they enter the box, from the top level: step limits around the
number of levels, and around what a ray needs, tell."""

import numpy as np
import pytest

import oracle
import synth
from oracle import voxel as ovox
from test_gpu_voxel import _compare, _levels_for, _render, hf  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("vz", [3, 5, 6, 7, 100])
def test_cameras_above_the_box(hf, vz):  # noqa: F811
    W, H = 400, 300
    h = np.full((H, W), 20)
    h[140:160, 140:160] = 255  # under the cameras
    h[140:160, 300:320] = 200
    h[10:60, 200:260] = 130
    cells = synth.pack_cells(h, 0, 0, 1).astype(np.uint32)
    box = -(-256 // vz) * vz
    cams = [synth.pose_to_camera(150.3, 150.2, z, yaw, pitch, 60, 40, 30)
            for z in (box - 0.5, box, box + 0.5, box + 4.0, box + 10.0, box + 30.0)
            for yaw, pitch in ((90.0, -4.0), (90.0, -15.0), (90.0, -25.0), (200.0, -10.0))]
    cams = synth.camera_array(cams)
    ctx = hf.hf_create(cells)
    try:
        hf.hf_voxel_build(ctx, 4, 4, vz)
        L = _levels_for(W // 4, H // 4, box // vz)
        g = ovox.Grid(cells, 4, 4, vz, L)
        for outer in [1, L - 1, L, L + 1] + list(range(12, 27, 2)) + [300]:
            got = _render(hf, ctx, cams, hf.make_voxel_opts(outer=outer, inner=4, far_dist=500.0))
            for i, cam in enumerate(cams):
                want = ovox.trace(g, cam["o"], oracle.ray_dirs(cam), far=500.0, outer=outer, inner=4)
                _compare(got[i], want, "vz %d outer %d cam %d" % (vz, outer, i))
    finally:
        hf.hf_destroy(ctx)
