"""The stored shadow bounds of large grids word for word (GPU only): builds of so
many groups of cells that a group's columns are not split over warps, whole
rounds are left out by level-5 nodes, and what still counts for a bound is carried
from round to round.  tests/test_gpu_sun_exact.py has the definition, restated
here on the GPU as its grids are small; the two are compared first."""

import numpy as np
import pytest

import synth
from test_gpu_sun_exact import _bounds, _definition, hf  # noqa: F401

pytestmark = pytest.mark.gpu


def _definition_gpu(cells, sun):
    import torch

    h0, h1, h2, _ = (torch.from_numpy(a.astype(np.int32)).cuda() for a in synth.unpack_cells(cells))
    top = torch.where(h1 > h0, h2, h0)
    x_major = abs(sun[0]) >= abs(sun[1])
    if not x_major:
        h0, top = h0.T.contiguous(), top.T.contiguous()
    lu, lv = (sun[0], sun[1]) if x_major else (sun[1], sun[0])
    lm, su = abs(lu), 1 if lu >= 0 else -1
    NV, NU = h0.shape
    cu = torch.arange(NU, device="cuda")
    cv = torch.arange(NV, device="cuda")

    def q(j):
        return (lv * j) // lm

    def column(a, k, none):  # a at major coordinate cu + su k, `none` past the grid
        u = cu + su * k
        return torch.where((u >= 0) & (u < NU), a[:, u.clamp(0, NU - 1)], none)

    def rows(a, r, none):  # a at minor coordinate cv + r
        v = cv + r
        return torch.where(((v >= 0) & (v < NV))[:, None], a[v.clamp(0, NV - 1)], none)

    def band(a, none, op, lo, hi):
        out = rows(a, lo, none)
        for r in range(lo + 1, hi + 1):
            out = op(out, rows(a, r, none))
        return out

    F = h0 * 256
    G = band(top, 0, torch.maximum, -1 if lv < 0 else 0, 1) * 256 + 1
    f_on = torch.ones_like(F, dtype=torch.bool)
    for k0 in range(1, 255 * lm // sun[2] + 40, 32):
        f_all = f_on.clone()
        for k in range(k0, k0 + 32):
            u = cu + su * k
            fl, fh = min(q(k - 1), q(k)), 1 + max(q(k - 1), q(k))
            gl, gh = min(q(k - 1), q(k + 1)), 1 + max(q(k - 1), q(k + 1))
            f_ok = ((u >= 0) & (u < NU))[None] & ((cv + fl >= 0) & (cv + fh < NV))[:, None]
            up, down = -(-256 * k * sun[2] // lm), 256 * (k - 1) * sun[2] // lm
            m = band(column(h0, k, 255), 255, torch.minimum, fl, fh)
            F = torch.where(f_on & f_ok, torch.maximum(F, m * 256 - up), F)
            # (a G term past the grid would be that of a top of 0, which raises nothing)
            t = band(column(top, k, 0), 0, torch.maximum, gl, gh)
            G = torch.maximum(G, t * 256 - down)
            f_all &= f_ok
        f_on = f_all
    out = (F | (G << 16)).cpu().numpy().view(np.uint32)
    return out if x_major else out.T


@pytest.mark.parametrize("W,H,pairs", [(2047, 1301, False), (1103, 2049, False), (1334, 1600, True)])
def test_large_builds_equal_their_definition(hf, W, H, pairs):  # noqa: F811
    groups = min(-(-W // 32) * -(-H // 4), -(-W // 64) * H)
    assert groups > 16384
    suns = [(321060, -321060, 262144), (-300000, 120000, 200000), (-110000, -380000, 300000),
            (37000, 401000, 100000), (401000, -37000, 100000), (700, 1000, 2000000)]
    small, _ = synth.make_grid(90, 70, seed=3, slab_frac=0.4, n_walls=9)
    for sun in suns[:4]:
        assert (_definition_gpu(small, sun) == _definition(small, sun)).all()
    cells, _ = synth.make_grid(W, H, seed=W + H, slab_frac=0.35, n_walls=W // 8)
    cells[: H // 3] = synth.pack_cells(20, 0, 0, 1)  # flat ground, where rounds are left out
    if pairs:
        cells = synth.pairify(cells)
    ctx = hf.hf_create_pairs(synth.encode_pairs(cells)) if pairs else hf.hf_create(cells)
    try:
        for sun in suns:
            got, want = _bounds(hf, ctx, sun), _definition_gpu(cells, sun)
            bad = np.argwhere(got != want)
            assert bad.size == 0, (sun, len(bad), bad[0], got[tuple(bad[0])], want[tuple(bad[0])])
    finally:
        hf.hf_destroy(ctx)
