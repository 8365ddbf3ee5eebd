"""Pyramids after edits of every small shape (GPU only): rectangles that start and
end inside their parents at the grid's corners, edges and middle, one cell, one
row, one column, and sizes around the ones where the last levels go to one block."""

import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hf():
    import paper_2608_17390_gb300 as m

    return m


@pytest.mark.parametrize("W,H,pairs", [(1999, 1501, False), (2, 4500, False), (4097, 3, False),
                                       (130, 4100, True), (1, 1, False), (257, 255, False)])
def test_pyramid_after_edits(hf, W, H, pairs):
    rng = np.random.default_rng(W + H)
    cells, _ = synth.make_grid(W, H, seed=W * 3 + H, slab_frac=0.4)
    if pairs:
        cells = synth.pairify(cells)
    ctx = hf.hf_create_pairs(synth.encode_pairs(cells)) if pairs else hf.hf_create(cells)
    sizes = [(1, 1), (61, 57), (64, 64), (65, 63), (2, 4100), (4096, 2), (90, 91), (1, 300), (700, 1),
             (2048, 3), (128, 64)]
    try:
        for k, (w, h) in enumerate(sizes):
            w, h = min(w, W), min(h, H)
            for place in range(3):
                x = [0, W - w, int(rng.integers(0, W - w + 1))][place]
                y = [0, H - h, int(rng.integers(0, H - h + 1))][place]
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
