"""Pyramids after edits whose lowest level is made in the block of the last ones,
or just not any more (GPU only): from 2048 to 4096 nodes on a level, in the grid's
corners and straddling parents, square and as thin as they can be."""

import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("W,H,pairs", [(1301, 901, False), (10000, 9, False), (6, 9000, True), (256, 256, False)])
def test_pyramid_after_edits(W, H, pairs):
    import paper_2608_17390_gb300 as hf

    rng = np.random.default_rng(W + H)
    cells, _ = synth.make_grid(W, H, seed=W * 5 + H, slab_frac=0.4)
    if pairs:
        cells = synth.pairify(cells)
    ctx = hf.hf_create_pairs(synth.encode_pairs(cells)) if pairs else hf.hf_create(cells)
    sizes = [(90, 90), (91, 92), (92, 92), (96, 96), (127, 129), (128, 128), (129, 129), (130, 128), (181, 90),
             (8192, 2), (8191, 3), (8190, 4), (4096, 4), (4094, 5), (2, 8191), (4, 4097), (2730, 6), (300, 300)]
    try:
        for k, (w, h) in enumerate(sizes):
            if pairs:
                w, h = min(w, h), max(w, h)
            w, h = min(w, W), min(h, H)
            for place in range(4):
                x = [0, W - w, int(rng.integers(0, W - w + 1)), (W - w) // 2 | 1 if W > w else 0][place]
                y = [0, H - h, int(rng.integers(0, H - h + 1)), (H - h) // 2][place]
                x = min(x, W - w)
                if pairs:
                    x, w = x // 2 * 2, max(2, w // 2 * 2)
                blk, _ = synth.make_grid(w, h, seed=100 * k + place, slab_frac=0.5)
                if pairs:
                    blk = synth.pairify(blk)
                hf.hf_edit(ctx, x, y, np.ascontiguousarray(blk))
                cells[y:y + h, x:x + w] = blk
            for lv, want in enumerate(oracle.pyramid(cells), 1):
                assert np.array_equal(hf.hf_read_pyramid(ctx, lv), want), (w, h, lv)
    finally:
        hf.hf_destroy(ctx)
