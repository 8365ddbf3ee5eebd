"""The march in beams against the oracle, bit for bit (GPU only): views whose
rays lie close enough, with enough samples in the grid, for the rules that pick
beams (which is checked): over odd, one-cell and paired grids in every direction, and
over the widest grids beside high columns, where a sample's rounding shows."""

import numpy as np
import pytest

import synth
from beamrule import march_in_beams, wide_views
from test_gpu_march import _gpu, hf  # noqa: F401
from test_gpu_march_edges import _check
from oracle import march

pytestmark = pytest.mark.gpu
S = 65536


def _compare(hf, cells, cams, steps, far, tile, texels=None):
    cams = synth.camera_array(cams)
    H, W = cells.shape
    assert not wide_views(W, H, cams, tile[0]).any() and march_in_beams(W, H, steps, far)
    ctx = hf.hf_create(cells) if texels is None else hf.hf_create_pairs(texels)
    try:
        got = _gpu(hf, ctx, cams, hf.make_march_opts(steps=steps, far_dist=far, tile_w=tile[0],
                                                     tile_h=tile[1]))
    finally:
        hf.hf_destroy(ctx)
    for i, c in enumerate(cams):
        _check(got[i], march.march_camera(cells, c, steps=steps, far=far), i)


@pytest.mark.parametrize("W,H,pairs", [(1, 1, False), (37, 53, False), (300, 9, False), (130, 97, True),
                                       (700, 613, False)])
@pytest.mark.parametrize("steps,part,tile", [(128, 1.0, (8, 4)), (1000, 3.0, (4, 32)), (113, 1.0, (32, 1)),
                                             (2000, 0.2, (8, 4)), (300, 0.0005, (16, 8))])
def test_close_rays(hf, W, H, pairs, steps, part, tile):  # noqa: F811
    far = part * max(W, H)
    rng = np.random.default_rng(W * H + steps)
    cells, _ = synth.make_grid(W, H, seed=W + H, slab_frac=0.4, n_walls=max(1, W // 10))
    if pairs:
        cells = synth.pairify(cells)
    cams = []
    for k in range(14):
        w, h = [(33, 5), (9, 41), (64, 3), (40, 30), (24, 24)][k % 5]
        x, y = rng.uniform(0.1, W - 0.1), rng.uniform(0.1, H - 0.1)
        if k % 3 == 0:
            x, y = float(int(x)), float(int(y))
        z = [0.0, 60.0, 125.0, 210.0, 400.0, 90.0, 3000.0][k % 7]
        hfov = 50.0 * w / max(tile[0], 32 // min(tile[0], 32)) * 0.035
        cams.append(synth.pose_to_camera(x, y, z, 51.0 * k, [-90, -45, -10, 0, -30, 20, -70][k % 7],
                                         min(hfov, 60.0), w, h))
    _compare(hf, cells, cams, steps, far, tile, synth.encode_pairs(cells) if pairs else None)


@pytest.mark.parametrize("wide", [True, False])
def test_starts_beside_boundaries_of_the_widest_grids(hf, wide):  # noqa: F811
    W, H = (16384, 24) if wide else (24, 16384)
    rng = np.random.default_rng(wide)
    h = np.full((H, W), 10, np.int64)
    at = [9568, 300, 4096, 8191, 16000]
    if wide:
        h[:, at] = 200
    else:
        h[at] = 200
    cells = synth.pack_cells(h, 0, 0, 1).astype(np.uint32)
    cams = []
    for k in range(40):
        side = (-1 if k % 2 else 1) * int([4, 1, 16, 32][k % 4])
        p = at[k % 5] + (k % 3 == 1) + side / S
        q = float(rng.integers(2, 22)) + [0.0, 0.3][k % 2]
        x, y = (p, q) if wide else (q, p)
        # the pixel scale of 1280 pixels in 75 degrees
        cams.append(synth.pose_to_camera(x, y, 100.0, 0.0 if k < 5 else 37.0 * k,
                                         -90 if k % 4 < 3 else -89.9, 8.2, 120, 80))
    _compare(hf, cells, cams, 128, 600.0, (8, 4))
    _compare(hf, cells, cams[::5], 1000, 600.0, (8, 4))
