"""The rule that tells wide views from those whose rays go in beams
(csrc/hf_rules.h), for tests that have to know which way a view goes."""

import numpy as np


def wide_views(W, H, cams, tile_w=8):
    """Per camera: whether a group of 32 of its pixels spans too much for a beam."""
    size = max(W, H)
    most = 0.06 if size <= 512 else 0.04 if size <= 4096 else 0.028
    gw = min(tile_w, 32)
    gh = 32 // gw
    f, r, u = (np.sqrt((cams[k].astype(float) ** 2).sum(1)) for k in "fru")
    return np.maximum(2 * gw * r, 2 * gh * u) > most * f


def share_of_wide(W, H, cams, tile_w=8):
    """The share of the batch's pixels that are in wide views."""
    px = cams["w"].astype(np.int64) * cams["h"]
    return px[wide_views(W, H, cams, tile_w)].sum() / px.sum()


def march_in_beams(W, H, steps, far):
    """Whether a march of close views takes beams."""
    return steps * min(1.0, max(W, H) / far) >= 112


def close_views(W, H, cams, tile_w=8):
    """The same cameras with their pixels brought together until none is wide."""
    cams = cams.copy()
    for i in range(len(cams)):
        one = cams[i:i + 1]
        while wide_views(W, H, one, tile_w)[0]:
            for k in "ru":
                one[k] = one[k] * 9 // 10
    assert not wide_views(W, H, cams, tile_w).any()
    return cams
