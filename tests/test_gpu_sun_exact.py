"""The stored shadow bounds word for word (GPU only).

tests/test_gpu_sun.py shows that the bounds are sound; here they equal their
definition, computed below with whole-array numpy from the cells: F the best
floor of a band less the rise up to the column, rounded down, G the highest top
of the wider band less the rise before it, rounded up, over the columns up to
the first round of 32 that holds one a bound cannot use.  Sizes around the
kernel's tiles (32 lanes, 4 or 2 cells a thread), grids with and without a
level 5, one row or one column, paired texels, and repairs.
"""

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu
S = 65536

SUNS = [(321060, -321060, 262144), (300000, 120000, 200000), (-300000, -290000, 250000),
        (-110000, -380000, 300000), (90000, 400000, 150000), (400000, 0, 300000),
        (0, -400000, 300000), (250000, 250000, 400000), (1000, -700, 2000000),
        (401000, 37000, 100000), (-37000, 401000, 100000)]
GRIDS = [(1, 1), (2, 40), (40, 2), (31, 33), (32, 64), (65, 127), (130, 47), (256, 300)]


@pytest.fixture(scope="module")
def hf():
    import torch

    import __graft_entry__

    __graft_entry__.build()
    assert torch.cuda.is_available()
    import paper_2608_17390_gb300 as m

    return m


def _definition(cells, sun):
    """F | G << 16 of every cell."""
    h0, h1, h2, _ = (a.astype(np.int64) for a in synth.unpack_cells(cells))
    top = np.where(h1 > h0, h2, h0)
    x_major = abs(sun[0]) >= abs(sun[1])
    if not x_major:
        h0, top = h0.T, top.T
    lu, lv = (sun[0], sun[1]) if x_major else (sun[1], sun[0])
    lm, su = abs(lu), 1 if lu >= 0 else -1
    NV, NU = h0.shape
    cu, cv = np.arange(NU)[None, :], np.arange(NV)[:, None]

    def q(j):
        return (lv * j) // lm

    def band(a, none, op, u, lo, hi):  # op over rows lo..hi (relative) of columns u, in the grid
        out = np.full((NV, NU), none, np.int64)
        for r in range(lo, hi + 1):
            rows = cv + r
            ok = (rows >= 0) & (rows < NV) & (u >= 0) & (u < NU)
            out = np.where(ok, op(out, a[np.clip(rows, 0, NV - 1), np.clip(u, 0, NU - 1)]), out)
        return out

    F = h0 * 256
    G = band(top, 0, np.maximum, cu, -1 if lv < 0 else 0, 1) * 256 + 1
    f_on = np.ones_like(F, bool)
    g_on = np.ones_like(F, bool)
    for k0 in range(1, 255 * lm // sun[2] + 40, 32):
        f_all, g_all = f_on.copy(), g_on.copy()
        for k in range(k0, k0 + 32):
            u = cu + su * k
            col = (u >= 0) & (u < NU)
            fl, fh = min(q(k - 1), q(k)), 1 + max(q(k - 1), q(k))
            gl, gh = min(q(k - 1), q(k + 1)), 1 + max(q(k - 1), q(k + 1))
            f_ok = col & (cv + fl >= 0) & (cv + fh < NV)
            g_ok = col & (cv + gh >= 0) & (cv + gl < NV)
            m = band(h0, 255, np.minimum, u, fl, fh)
            t = band(top, 0, np.maximum, u, gl, gh)
            up, down = -(-256 * k * sun[2] // lm), 256 * (k - 1) * sun[2] // lm
            F = np.where(f_on & f_ok, np.maximum(F, m * 256 - up), F)
            G = np.where(g_on & g_ok, np.maximum(G, t * 256 - down), G)
            f_all &= f_ok
            g_all &= g_ok
        f_on, g_on = f_all, g_all
    out = (F | (G << 16)).astype(np.uint32)
    return out if x_major else out.T


def _bounds(hf, ctx, sun):
    cam = synth.camera_array([synth.ray_camera((5, 7, S * 250), (1000, 1300, -9000))])
    hf.hf_render(ctx, cam, hf.alloc_outputs(cam, shadows=True),
                 hf.make_opts(flags=hf.HF_SHADOWS | hf.HF_SYNC, sun=sun))
    return hf.hf_read_sun_bounds(ctx)[0]


@pytest.mark.parametrize("W,H", GRIDS)
@pytest.mark.parametrize("pairs", (False, True))
def test_bounds_equal_their_definition(hf, W, H, pairs):
    if pairs and W % 2:
        pytest.skip("paired texels need an even width")
    cells, _ = synth.make_grid(W, H, seed=W + 7 * H, slab_frac=0.35, n_walls=max(1, W // 12))
    if pairs:
        cells = synth.pairify(cells)
    ctx = hf.hf_create_pairs(synth.encode_pairs(cells)) if pairs else hf.hf_create(cells)
    try:
        for sun in SUNS:
            got, want = _bounds(hf, ctx, sun), _definition(cells, sun)
            bad = np.argwhere(got != want)
            assert bad.size == 0, (sun, len(bad), bad[0], got[tuple(bad[0])], want[tuple(bad[0])])
        rng = np.random.default_rng(1)
        for sun in SUNS[:5]:  # a repair after an edit
            _bounds(hf, ctx, sun)
            w, h = int(rng.integers(1, min(W, 20) + 1)), int(rng.integers(1, min(H, 20) + 1))
            x, y = int(rng.integers(0, W - w + 1)), int(rng.integers(0, H - h + 1))
            if pairs:
                x, w = x & ~1, min((w + 1) & ~1, W - (x & ~1))
            blk = cells[y:y + h, x:x + w] & np.uint32(0xFF000000)
            cells[y:y + h, x:x + w] = blk | np.uint32(rng.integers(0, 250))
            hf.hf_edit(ctx, x, y, np.ascontiguousarray(cells[y:y + h, x:x + w]))
            got, want = hf.hf_read_sun_bounds(ctx)[0], _definition(cells, sun)
            assert (got == want).all(), (sun, np.argwhere(got != want)[:3])
    finally:
        hf.hf_destroy(ctx)
