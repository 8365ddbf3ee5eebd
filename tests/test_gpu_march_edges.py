"""The marcher's choice of samples at its edges (GPU only), bit for bit against
the oracle, which takes every sample: rays along an axis and in every octant,
vertical, level, rising and from height 0, sample spacings from a fraction of a
cell to many times the grid, odd images and tiles, odd and one-cell grids, caves
and walls, paired texels."""

import numpy as np
import pytest

import synth
from oracle import march
from test_gpu_march import _gpu, hf  # noqa: F401

pytestmark = pytest.mark.gpu
S = 65536


def _check(got, ref, what):
    for k in ("hit_cell", "layer"):
        assert np.array_equal(got[k], ref[k]), (what, k)
    assert np.array_equal(got["depth"].view(np.uint32), ref["depth"].view(np.uint32)), what


@pytest.mark.parametrize("wide", [True, False])
@pytest.mark.parametrize("W,H,pairs", [(1, 1, False), (37, 53, False), (300, 9, False), (130, 97, True)])
@pytest.mark.parametrize("steps,far,tile", [(128, 600.0, (8, 4)), (1000, 90.0, (4, 32)), (7, 5000.0, (32, 1)),
                                            (64, 0.05, (16, 8))])
def test_samples_around_the_beams(hf, W, H, pairs, steps, far, tile, wide):
    rng = np.random.default_rng(W * H + steps)
    cells, _ = synth.make_grid(W, H, seed=W + H, slab_frac=0.4, n_walls=max(1, W // 10))
    if pairs:
        cells = synth.pairify(cells)
    cams = []
    for k, (w, h) in enumerate([(1, 1), (33, 5), (9, 41), (64, 3), (40, 30), (40, 30), (24, 24)]):
        x, y = rng.uniform(0.1, W - 0.1), rng.uniform(0.1, H - 0.1)
        z = [0.0, 60.0, 125.0, 210.0, 400.0, 90.0, 3000.0][k]
        hfov = 60 if max(w, h) < 30 or w >= h else 10
        if not wide:  # (rays close enough for beams)
            hfov = min(0.09 * w / max(min(tile[0], 32), 32 // min(tile[0], 32)) * 45, 60)
        cams.append(synth.pose_to_camera(x, y, z, 51.0 * k, [-90, -45, -10, 0, -30, 20, -70][k], hfov, w, h))
    for g in range(60):
        o = [int(rng.integers(0, W * S)), int(rng.integers(0, H * S)), int(rng.integers(0, 250 * S))]
        if g % 2:
            o = [v // S * S for v in o]
        d = [int(v) * [1, 1000, 300000][g % 3] for v in rng.integers(-3, 4, 3)]
        cams.append(synth.ray_camera(o, d if any(d) else (0, 0, -5)))
    cams = synth.camera_array(cams)
    ctx = hf.hf_create_pairs(synth.encode_pairs(cells)) if pairs else hf.hf_create(cells)
    try:
        got = _gpu(hf, ctx, cams, hf.make_march_opts(steps=steps, far_dist=far, tile_w=tile[0],
                                                     tile_h=tile[1]))
        for i, c in enumerate(cams):
            _check(got[i], march.march_camera(cells, c, steps=steps, far=far), i)
    finally:
        hf.hf_destroy(ctx)
