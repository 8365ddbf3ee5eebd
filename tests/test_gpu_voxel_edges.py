"""RayVoxel at the sizes where its kernels can go wrong (GPU only), against the
oracle: occupancy words for every width of layer mask, grids around the 8-voxel
tiles and repairs across their edges; rays along an axis, on voxel planes and in
every octant, images that fill no 8 x 4 tile, more levels than the grid needs."""

import numpy as np
import pytest

import oracle
import synth
from oracle import voxel as ovox
from test_gpu_voxel import _check_words, _compare, _levels_for, _rand_grid, _render, hf  # noqa: F401

pytestmark = pytest.mark.gpu
S = 65536


@pytest.mark.parametrize("v", [(1, 1, 1), (4, 2, 2), (2, 3, 3), (1, 2, 4), (5, 1, 9), (64, 64, 256)])
@pytest.mark.parametrize("W,H", [(1, 1), (8, 31), (33, 17), (68, 64)])
def test_words_around_tiles(hf, v, W, H):
    rng = np.random.default_rng(W * 100 + H + sum(v))
    cells = _rand_grid(rng, W, H, hmax=255)
    ctx = hf.hf_create(cells)
    try:
        L = _levels_for(-(-W // v[0]), -(-H // v[1]), -(-256 // v[2]))
        hf.hf_voxel_build(ctx, *v)
        _check_words(hf, ctx, cells, v, L, "build")
        hf.hf_voxel_build(ctx, *v)  # again, in the same memory
        for _ in range(6):
            w, h = int(rng.integers(1, min(W, 12) + 1)), int(rng.integers(1, min(H, 12) + 1))
            x, y = int(rng.integers(0, W - w + 1)), int(rng.integers(0, H - h + 1))
            blk = _rand_grid(rng, w, h, hmax=30)
            hf.hf_edit(ctx, x, y, blk)
            cells[y:y + h, x:x + w] = blk
            _check_words(hf, ctx, cells, v, L, "repair")
    finally:
        hf.hf_destroy(ctx)


@pytest.mark.parametrize("v,levels", [((4, 8, 2), 0), ((1, 1, 1), 0), ((3, 4, 2), 0), ((8, 4, 16), 9),
                                      ((2, 5, 3), 8)])
def test_rays_along_planes_and_axes(hf, v, levels):
    rng = np.random.default_rng(sum(v))
    W, H = 45, 39
    cells = _rand_grid(rng, W, H, hmax=60)
    rays = []
    for g in range(160):
        q = [S, 4 * S, S // 2, 1][g % 4]
        o = [int(rng.integers(0, n * S)) // q * q for n in (W, H, 200)]
        d = [int(x) * [1, 1000, 300000][g % 3] for x in rng.integers(-3, 4, 3)]
        rays.append(synth.ray_camera(o, d if any(d) else (0, 0, -1)))
    views = [synth.pose_to_camera(W / 2, H / 3, 120.0, 40.0 * k, -30.0, 70, w, h)
             for k, (w, h) in enumerate([(1, 1), (7, 3), (33, 5), (9, 41), (64, 2)])]
    cams = synth.camera_array(rays + views)
    ctx = hf.hf_create(cells)
    try:
        hf.hf_voxel_build(ctx, *v, levels)
        L = levels or _levels_for(-(-W // v[0]), -(-H // v[1]), -(-256 // v[2]))
        g = ovox.Grid(cells, *v, L)
        got = _render(hf, ctx, cams, hf.make_voxel_opts(inner=3))
        for i, cam in enumerate(cams):
            want = ovox.trace(g, cam["o"], oracle.ray_dirs(cam), inner=3)
            _compare(got[i], want, "cam %d" % i)
    finally:
        hf.hf_destroy(ctx)
