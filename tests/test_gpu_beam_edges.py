"""Beams of close rays where they can go wrong (GPU only), every pixel against the
oracle: odd and one-row grids, caves and walls, cameras in every octant, level,
rising and falling, on cell boundaries and the grid's edge, tiles of every
kind, all pyramid limits, and batches that mix close and far-apart rays."""

import numpy as np
import pytest

import oracle
import synth
from hfcheck import compare, gpu_render

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hf():
    import paper_2608_17390_gb300 as m

    return m


@pytest.mark.parametrize("W,H,pairs", [(37, 53, False), (301, 9, False), (2, 200, False),
                                       (130, 97, True), (640, 500, False)])
@pytest.mark.parametrize("tile,mip", [((0, 0), 6), ((4, 64), 5), ((8, 16), 0), ((32, 1), 2), ((2, 16), 1)])
def test_close_rays_equal_the_oracle(hf, W, H, pairs, tile, mip):
    cells, _ = synth.make_grid(W, H, seed=W + 7 * H, slab_frac=0.4, n_walls=max(1, W // 8))
    if pairs:
        cells = synth.pairify(cells)
    rng = np.random.default_rng(W + H)
    cams = []
    for k in range(16):
        x, y = rng.uniform(0, W), rng.uniform(0, H)
        if k % 3 == 0:
            x, y = float(int(x)), float(int(y))
        z = [2.0, 60.0, 140.0, 254.0, 300.0][k % 5]
        cams.append(synth.pose_to_camera(x, y, z, 22.5 * k + (k % 4), [0, -20, -60, 8, -89][k % 5], 6.0,
                                         [65, 96, 127][k % 3], [33, 70][k % 2]))
    if tile == (0, 0):  # a few rays far apart
        cams.append(synth.pose_to_camera(W / 2, H / 2, 200.0, 10.0, -40.0, 80.0, 33, 17))
    cams = synth.camera_array(cams)
    ctx = hf.hf_create_pairs(synth.encode_pairs(cells)) if pairs else hf.hf_create(cells)
    try:
        for shadows in (False, True):
            opts = hf.make_opts(flags=hf.HF_SHADOWS if shadows else 0, tile_w=tile[0], tile_h=tile[1],
                                mip_start=mip)
            got = gpu_render(hf, ctx, cams, shadows=shadows, opts=opts)
            for i, c in enumerate(cams):
                want = oracle.render(cells, c, shadows=shadows)
                compare(got[i], want, shadows=shadows, what="%dx%d cam %d" % (W, H, i))
    finally:
        hf.hf_destroy(ctx)
