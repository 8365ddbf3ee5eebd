"""The views of the parity tests with their rays close together (GPU only), so that
the kernels of beams trace them: random worlds with random suns and edits between
shadowed renders, plain and paired texels; every climb limit and tile shape;
hand-made edge cases; cameras at node tops, in caves and on corners; straight
down; the largest batch; and the largest grid with cameras at the limits, before
and after edits.  Every pixel against the oracle."""

import os

import numpy as np
import pytest

import oracle
import synth
from beamrule import close_views, wide_views
from hfcheck import compare, gpu_render
from test_gpu_fullsize import _max_world
from test_gpu_parity import _rand_grid
from test_gpu_random import SHAPES, _cams, _cells, _sun, hf  # noqa: F401

pytestmark = pytest.mark.gpu
NT = os.cpu_count() or 4


@pytest.mark.parametrize("k", range(len(SHAPES) * 6))
def test_random_worlds_suns_and_edits(hf, k):  # noqa: F811
    rng = np.random.default_rng(9100 + k)
    W, H = SHAPES[k % len(SHAPES)]
    pairs = W % 2 == 0 and k % 4 == 1
    cells = _cells(rng, W, H) & np.uint32(0x07FFFFFF)
    if pairs:
        cells = synth.pairify(cells)
    sun = _sun(rng, k)
    cams = close_views(W, H, _cams(rng, W, H, 7))
    opts = hf.make_opts(flags=hf.HF_SHADOWS, sun=sun,
                        mip_start=int(rng.integers(0, 8)) if k % 3 else hf.HF_MIP_AUTO)
    ctx = hf.hf_create_pairs(synth.encode_pairs(cells)) if pairs else hf.hf_create(cells)
    try:
        for step in range(3):
            g = gpu_render(hf, ctx, cams, shadows=True, opts=opts)
            for i, c in enumerate(cams):
                compare(g[i], oracle.render(cells, c, shadows=True, sun=sun, nthreads=NT), shadows=True,
                        what="world %dx%d sun %s step %d cam %d" % (W, H, sun, step, i))
            ew, eh = min(int(rng.integers(1, W + 1)), 24), min(int(rng.integers(1, H + 1)), 24)
            x0, y0 = int(rng.integers(0, W - ew + 1)), int(rng.integers(0, H - eh + 1))
            if pairs:
                x0, ew = x0 // 2 * 2, max(2, ew // 2 * 2)
            blk = _cells(rng, ew, eh) & np.uint32(0x07FFFFFF)
            if pairs:
                blk = synth.pairify(blk)
            hf.hf_edit(ctx, x0, y0, blk)
            cells[y0:y0 + eh, x0:x0 + ew] = blk
    finally:
        hf.hf_destroy(ctx)


@pytest.mark.parametrize("mip", [0, 1, 2, 4, 6, 8, 30])
@pytest.mark.parametrize("tile", [(8, 4), (32, 1), (4, 8), (16, 4), (16, 16), (1, 64), (256, 1)])
def test_every_climb_limit_and_tile_shape(hf, mip, tile):  # noqa: F811
    cells = synth.config_c1()["cells"]
    H, W = cells.shape
    cams = close_views(W, H, synth.camera_array(
        [synth.pose_to_camera(128.5, 16.5, 140.0, 0.0, -35.0, 60.0, 80, 60),
         synth.pose_to_camera(40.25, 200.75, 60.0, 130.0, -8.0, 60.0, 61, 45),
         synth.pose_to_camera(200.0, 100.0, 250.0, 250.0, -80.0, 60.0, 33, 70)]), tile[0])
    ctx = hf.hf_create(cells)
    try:
        g = gpu_render(hf, ctx, cams, shadows=True,
                       opts=hf.make_opts(tile_w=tile[0], tile_h=tile[1], mip_start=mip, flags=hf.HF_SHADOWS))
        for i, c in enumerate(cams):
            compare(g[i], oracle.render(cells, c, shadows=True), shadows=True, what="mip %d tile %s" % (mip, tile))
    finally:
        hf.hf_destroy(ctx)


def test_edge_cases(hf):  # noqa: F811
    rng = np.random.default_rng(7)
    P = synth.pose_to_camera
    odd = [(18.5, 14.5, 40.0, 10, -90), (0.0, 28.99, 10.0, 135, -5), (36.99, 0.0, 2.0, 300, 20)]
    cases = [
        (np.array([[synth.pack_cells(3, 5, 9, 2)]], np.uint32),
         [P(0.5, 0.5, 7.0, 0, -90, 60, 3, 3), P(0.0, 0.0, 4.0, 45, -10, 90, 5, 4)]),
        (_rand_grid(rng, 37, 29, 30), [P(*p, 80, w, h) for p in odd for w, h in ((33, 17), (31, 9), (64, 3))]),
        (_rand_grid(rng, 16384, 16, 40), [P(16383.9, 8.0, 30.0, 270, -1, 20, 97, 5), P(0.1, 8.0, 30.0, 90, -1, 20, 97, 5),
                                          P(8192.0, 8.0, 30.0, 90, -0.2, 20, 97, 5)]),
        (_rand_grid(rng, 16, 16384, 40), [P(8.0, 16383.9, 30.0, 180, -1, 20, 97, 5), P(8.0, 0.1, 30.0, 0, -1, 20, 97, 5),
                                          P(8.0, 8192.0, 30.0, 0, -0.2, 20, 97, 5)]),
        (_rand_grid(rng, 37, 29, 30), [P(18.5, 14.5, 40.0, 30, -30, 120, int(hf.HF_MAX_DIM), 2)]),
        (np.zeros((8, 8), np.uint32), [P(4.0, 4.0, 3.0, 0, -90, 90, 7, 7), P(8.0 - 1 / 65536, 0.0, 0.0, 10, -45, 90, 7, 7)])]
    for cells, poses in cases:
        H, W = cells.shape
        cams = close_views(W, H, synth.camera_array(poses))
        ctx = hf.hf_create(cells)
        try:
            g = gpu_render(hf, ctx, cams, shadows=True, opts=hf.make_opts(flags=hf.HF_SHADOWS))
            for i, c in enumerate(cams):
                compare(g[i], oracle.render(cells, c, shadows=True), shadows=True, what="edge %s cam %d" % (cells.shape, i))
        finally:
            hf.hf_destroy(ctx)


def test_cameras_at_node_tops_in_caves_and_straight_down(hf):  # noqa: F811
    rng = np.random.default_rng(2024)
    cells = _rand_grid(rng, 96, 80, hmax=40)
    levels = oracle.pyramid(cells)
    h0, h1, h2, _ = (a.astype(int) for a in synth.unpack_cells(cells))
    poses = []
    for k, (x, y) in enumerate([(40.0, 33.0), (10.5, 70.25), (77.0, 12.0)]):
        cx, cy = int(x), int(y)
        tops = [h2[cy, cx] if h1[cy, cx] > h0[cy, cx] else h0[cy, cx]]
        tops += [int((lv[cy >> (i + 1), cx >> (i + 1)] >> 16) & 0xFF) for i, lv in enumerate(levels)]
        for lvl in (0, 2, 4):
            for dz in (0.0, 1.0 / 65536):
                poses.append(synth.pose_to_camera(x, y, tops[lvl] + dz, 97.0 * k + 31 * lvl, -20.0 + 10 * lvl, 80, 23, 11))
    cave = np.argwhere(h1 > h0 + 1)[0]
    mid = (h0[tuple(cave)] + h1[tuple(cave)]) / 2.0
    for yaw, pitch in ((200, 5), (20, -30), (110, 60), (0, 89)):
        poses.append(synth.pose_to_camera(cave[1] + 0.5, cave[0] + 0.5, mid, yaw, pitch, 90, 31, 9))
    poses.append(synth.pose_to_camera(0.0, 0.0, 50.0, 225, -30, 70, 27, 13))
    poses.append(synth.pose_to_camera(48.0, 40.0, 45.0, 225, -45, 70, 27, 13))
    # odd sizes put a pixel on the axis: a vertical ray among the beam's
    poses += [synth.pose_to_camera(x, y, 90.0, 0, -90, 60, 9, 9) for x, y in ((8.0, 8.0), (30.5, 7.25), (95.9, 79.9))]
    cams = close_views(96, 80, synth.camera_array(poses))
    ctx = hf.hf_create(cells)
    try:
        orc = [oracle.render(cells, c, shadows=True) for c in cams]
        for mip in (0, 1, 3, 5, 7):
            g = gpu_render(hf, ctx, cams, shadows=True, opts=hf.make_opts(mip_start=mip, flags=hf.HF_SHADOWS))
            for i in range(len(cams)):
                compare(g[i], orc[i], shadows=True, what="cam %d mip %d" % (i, mip))
    finally:
        hf.hf_destroy(ctx)


def test_largest_batch(hf):  # noqa: F811
    cells = synth.config_c1()["cells"]
    H, W = cells.shape
    rng = np.random.default_rng(3)
    n = int(hf.HF_MAX_CAMERAS)
    cams = close_views(W, H, synth.camera_array(
        [synth.pose_to_camera(float(rng.uniform(1, 255)), float(rng.uniform(1, 255)), float(rng.uniform(20, 250)),
                              float(rng.uniform(0, 360)), float(rng.uniform(-89, 10)), float(rng.uniform(20, 40)), 8, 4)
         for _ in range(n)]))
    ctx = hf.hf_create(cells)
    try:
        g = gpu_render(hf, ctx, cams, shadows=True)
        p = gpu_render(hf, ctx, cams, shadows=True, opts=hf.make_opts(flags=hf.HF_SHADOWS | hf.HF_PLAIN))
        for i in range(n):
            for k in g[i]:
                assert np.array_equal(g[i][k], p[i][k]), (i, k)
        for i in range(0, n, 61):
            compare(g[i], oracle.render(cells, cams[i], shadows=True), shadows=True, what="camera %d" % i)
    finally:
        hf.hf_destroy(ctx)


def test_largest_grid_and_edits(hf):  # noqa: F811
    """Rays across the whole of 16384 x 16384 cells, from the greatest altitude, from
    the far corner, and where cells change: before and after a strip across the
    2^27-cell index and a crater in the far corner."""
    cells = _max_world(seed=12)
    P = synth.pose_to_camera
    cams = close_views(16384, 16384, synth.camera_array(
        [P(0.5, 0.5, 150.0, 45, -0.06, 20, 96, 12), P(8192.5, 8192.5, 4095.0, 0, -90, 120, 63, 63),
         P(8192.5, 8192.5, 4095.0, 70, -30, 120, 64, 64), P(16383.5, 16383.5, 140.0, 225, 0.5, 90, 97, 33),
         P(8192.5, 8150.5, 300.0, 0, -20, 90, 64, 32), P(16300.5, 16250.5, 120.0, 30, -30, 90, 48, 24)]))
    assert not wide_views(16384, 16384, cams).any()
    rng = np.random.default_rng(13)
    strip = synth.pack_cells(rng.integers(0, 150, (40, 16384)), 0, 0, rng.integers(0, 8, (40, 16384)))
    ctx = hf.hf_create(cells)
    try:
        for edited in (False, True):
            if edited:
                hf.hf_edit(ctx, 0, 8180, strip)
                cells[8180:8220, :] = strip
                x0, y0, blk = synth.crater_edit(cells, 16330, 16340)
                hf.hf_edit(ctx, x0, y0, blk)
                cells[y0:y0 + blk.shape[0], x0:x0 + blk.shape[1]] = blk
            g = gpu_render(hf, ctx, cams, shadows=True)
            for i, c in enumerate(cams):
                compare(g[i], oracle.render(cells, c, shadows=True, nthreads=NT), shadows=True,
                        what="camera %d edited %d" % (i, edited))
    finally:
        hf.hf_destroy(ctx)
