"""Batches of close and wide views (GPU only), in any order: the wide ones' rays go
each by itself in the kernel of the beams, at the head of the launch.  Every
view has to equal the oracle, and every way to launch the batch the others."""

import numpy as np
import pytest

import oracle
import synth
from beamrule import march_in_beams, share_of_wide, wide_views
from hfcheck import compare, gpu_render
from oracle import march
from test_gpu_march import _gpu, hf  # noqa: F401
from test_gpu_march_edges import _check

pytestmark = pytest.mark.gpu


def _views(W, H, order, n_wide, wide_px, seed):
    rng = np.random.default_rng(seed)
    cams = []
    for k in range(len(order) * 2):
        x, y, z = rng.uniform(0, W), rng.uniform(0, H), [3.0, 90.0, 200.0, 300.0][k % 4]
        if k % 5 == 0:
            x, y = float(int(x)), float(int(y))
        pose = (x, y, z, 47.0 * k, [-10, -40, -90, 5][k % 4])
        if order[k % len(order)] == "w" and n_wide:
            n_wide -= 1
            cams.append(synth.pose_to_camera(*pose, 70.0, *wide_px))
        else:
            cams.append(synth.pose_to_camera(*pose, 9.0, [97, 128][k % 2], [70, 65][k % 2]))
    return synth.camera_array(cams)


@pytest.mark.parametrize("W,H,pairs", [(97, 60, False), (700, 333, False), (130, 1000, True), (4200, 20, False)])
@pytest.mark.parametrize("order", ["w...", "...w", ".w.w"])
def test_traced(hf, W, H, pairs, order):  # noqa: F811
    cells, _ = synth.make_grid(W, H, seed=W + H, slab_frac=0.4, n_walls=W // 10)
    if pairs:
        cells = synth.pairify(cells)
    cams = _views(W, H, order, 4, (41, 30), W)
    if W > 4096:  # (a longer world allows less)
        cams["r"] //= 2
        cams["u"] //= 2
    wide = wide_views(W, H, cams)
    assert wide.any() and not wide.all() and 0 < share_of_wide(W, H, cams) <= 1 / 4
    ctx = hf.hf_create_pairs(synth.encode_pairs(cells)) if pairs else hf.hf_create(cells)
    try:
        for flags in (0, hf.HF_SHADOWS, hf.HF_SHADOWS | hf.HF_NOGRAPH, hf.HF_SHADOWS | hf.HF_PLAIN):
            sh = bool(flags & hf.HF_SHADOWS)
            got = gpu_render(hf, ctx, cams, shadows=sh, opts=hf.make_opts(flags=flags))
            for i, c in enumerate(cams):
                compare(got[i], oracle.render(cells, c, shadows=sh), shadows=sh, what="cam %d %d" % (i, flags))
        outs = hf.alloc_outputs(cams, shadows=True)
        hf.hf_render_noalloc(ctx, cams, outs, hf.make_opts(flags=hf.HF_SHADOWS | hf.HF_SYNC))
        for o, g in zip(outs, got):
            for k in o:
                a = o[k].cpu().numpy()
                assert np.array_equal(a.view(np.uint8), g[k].view(np.uint8)), k
    finally:
        hf.hf_destroy(ctx)


@pytest.mark.parametrize("W,H", [(97, 60), (700, 333)])
@pytest.mark.parametrize("order", ["w...", "...w"])
def test_marched(hf, W, H, order):  # noqa: F811
    cells, _ = synth.make_grid(W, H, seed=W + H, slab_frac=0.4, n_walls=W // 10)
    cams = _views(W, H, order, 1, (24, 16), W)
    assert 0 < share_of_wide(W, H, cams) <= 1 / 32
    ctx = hf.hf_create(cells)
    try:
        far = float(max(W, H))
        assert march_in_beams(W, H, 128, far)
        got = _gpu(hf, ctx, cams, hf.make_march_opts(steps=128, far_dist=far))
        for i, c in enumerate(cams):
            _check(got[i], march.march_camera(cells, c, steps=128, far=far), i)
    finally:
        hf.hf_destroy(ctx)
