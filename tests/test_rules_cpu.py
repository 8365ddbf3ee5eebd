"""The rules that pick a render's launch from its cameras (csrc/hf_rules.h), on
the CPU."""

import ctypes
import os
import subprocess

import numpy as np
import pytest

import synth

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SHIM = r"""
#include "hf_rules.h"
extern "C" void tile(const hf_camera *c, uint32_t n, int beams, uint64_t warps, uint32_t flags, uint32_t *t) {
    hf::default_tile(c, n, beams, warps, flags, t[0], t[1]);
}
extern "C" int pay(int32_t W, int32_t H, int32_t steps, float far_dist) { return hf::march_beams_pay(W, H, steps, far_dist); }
extern "C" int wide(int32_t W, int32_t H, const hf_camera *c, uint32_t tw) { return hf::view_wide(W, H, *c, tw); }
extern "C" int fit(int32_t W, int32_t H, const hf_camera *c, uint32_t n, uint32_t tw, uint32_t share) {
    uint8_t wide[64];
    return hf::beams_fit(W, H, c, n, tw, share, wide);
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("rules")
    (d / "shim.cpp").write_text(SHIM)
    so = str(d / "rules.so")
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", os.path.join(ROOT, "include"),
                           "-I", os.path.join(ROOT, "paper_2608_17390_gb300", "csrc"),
                           str(d / "shim.cpp"), "-o", so])
    return ctypes.CDLL(so)


def _cams(w, h, n):
    return np.repeat(synth.camera_array([((0, 0, 0), (1 << 19, 0, 0), (0, 9, 0), (0, 0, 9), w, h)]), n)


def _tile(lib, cams, warps=3648, beams=True, flags=0):
    t = (ctypes.c_uint32 * 2)()
    lib.tile(ctypes.c_void_p(cams.ctypes.data), len(cams), int(beams), ctypes.c_uint64(warps), flags, t)
    return tuple(t)


@pytest.mark.parametrize("w,h,n,want", [
    (320, 240, 1, (8, 4)), (1280, 720, 1, (4, 8)), (1920, 1080, 1, (4, 16)), (3840, 2160, 1, (4, 32)),
    (1920, 1080, 100, (4, 32)), (640, 360, 100, (4, 32)), (16384, 16384, 1, (4, 32)),
    # images lower than the tiles, or a little higher than a number of them
    (2048, 1, 4096, (8, 4)), (2048, 2, 4000, (8, 4)), (3840, 9, 100, (8, 4)), (3840, 9, 4000, (8, 4)),
    (3840, 8, 4000, (4, 8)), (1024, 17, 4000, (8, 4)), (1024, 40, 4000, (4, 8)), (1024, 32, 4000, (4, 32)),
    (1, 1, 4096, (8, 4)), (2, 512, 4096, (4, 16))])
def test_default_tile(lib, w, h, n, want):
    assert _tile(lib, _cams(w, h, n)) == want
    assert _tile(lib, _cams(w, h, n), beams=False) == (8, 4)
    assert _tile(lib, _cams(w, h, n), flags=64 | 128 | 256) == (8, 4)


def test_default_tile_makes_no_more_groups(lib):
    rng = np.random.default_rng(2)
    for _ in range(300):
        cams = np.concatenate([_cams(*(int(2.0 ** rng.uniform(0, 13)) for _ in range(2)), int(rng.integers(1, 40)))
                               for _ in range(3)])
        tw, th = _tile(lib, cams)
        w, h = cams["w"].astype(np.int64), cams["h"].astype(np.int64)
        wide = (-(-w // 8) * -(-h // 4)).sum()
        if tw == 4:
            assert (-(-w // 4) * -(-h // 8)).sum() <= wide * 33 / 32
            assert (-(-w // 4) * -(-h // th)).sum() * (th // 8) <= (-(-w // 4) * -(-h // 8)).sum() * 9 / 8


def test_a_batch_refused_in_8_by_4_tiles_stays_refused(lib):
    """2^32 tiles of 8 x 4 are one too many; taller tiles would make them fewer."""
    assert _tile(lib, _cams(16384, 16384, 512)) == (8, 4)
    assert _tile(lib, _cams(16384, 16384, 511)) == (4, 32)


@pytest.mark.parametrize("W,H,most", [(512, 200, 0.06), (513, 4, 0.04), (30, 4096, 0.04), (4097, 2, 0.028)])
@pytest.mark.parametrize("tw", [1, 4, 8, 32, 256])
def test_view_wide(lib, W, H, most, tw):
    """A group of 32 pixels that spans more than `most` radians; pixels of 2 / f."""
    gw = min(tw, 32)
    long = max(gw, 32 // gw)
    for span, want in ((0.98 * most, False), (1.02 * most, True)):
        f = int(round(2 * long * 999 / span))
        cams = synth.camera_array([((0, 0, 0), (0, f, 0), (999, 0, 0), (0, 0, 999), 64, 48)])
        assert bool(lib.wide(W, H, ctypes.c_void_p(cams.ctypes.data), tw)) == want


def test_share_of_wide_views(lib):
    """Wide pixels: up to a quarter of a traced batch, one in 32 of a marched one."""
    f = 2 * 8 * 999
    narrow = synth.camera_array([((0, 0, 0), (0, f * 100, 0), (999, 0, 0), (0, 0, 999), 64, 32)])
    wide = synth.camera_array([((0, 0, 0), (0, f, 0), (999, 0, 0), (0, 0, 999), 64, 32)])
    for share in (4, 32):
        for k, want in ((share - 1, True), (share - 2, False)):
            cams = np.concatenate([wide, np.repeat(narrow, k)])
            fit = lib.fit(300, 300, ctypes.c_void_p(cams.ctypes.data), len(cams), 8, share)
            assert bool(fit) == want, (share, k)


@pytest.mark.parametrize("W,H,steps,far,want", [
    (2048, 16384, 112, 600.0, True), (2048, 16384, 111, 600.0, False), (300, 2, 128, 300.0, True),
    (300, 200, 223, 600.0, False), (300, 200, 224, 600.0, True), (1, 1, 65536, 600.0, False),
    (1, 1, 112, 0.5, True), (16384, 16384, 1, 1e30, False)])
def test_march_beams_pay(lib, W, H, steps, far, want):
    assert bool(lib.pay(W, H, steps, ctypes.c_float(far))) == want
