"""The tile that a render takes when its sides are left at 0 depends on the size
of the batch; every choice gives the pixels of 8 x 4 tiles."""
import pytest

torch = pytest.importorskip("torch")

import paper_2608_17390_gb300 as hf
import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("w,h,n", [(33, 17, 1), (1201, 801, 1), (1921, 1083, 1), (4001, 2163, 1),
                                   (1283, 717, 2), (641, 363, 40)])
@pytest.mark.parametrize("shadows", [False, True])
def test_default_tile_equals_8x4(w, h, n, shadows):
    cells, _ = synth.make_grid(160, 96, seed=11, slab_frac=0.4, n_walls=12)
    ctx = hf.hf_create(cells)
    cams = synth.camera_array([synth.pose_to_camera(60.3 + i, 40.7, 130.0 + i, 31.0 + 9 * i, -24.0,
                                                    70.0, w, h) for i in range(n)])
    flags = hf.HF_SHADOWS | hf.HF_SYNC if shadows else hf.HF_SYNC
    a = hf.alloc_outputs(cams, shadows=shadows)
    b = hf.alloc_outputs(cams, shadows=shadows)
    hf.hf_render(ctx, cams, a, hf.make_opts(flags=flags))
    hf.hf_render(ctx, cams, b, hf.make_opts(flags=flags, tile_w=8, tile_h=4))
    for x, y in zip(a, b):
        for k in x:
            assert torch.equal(x[k], y[k]), k
    hf.hf_destroy(ctx)
