"""The rays that no beam takes (vertical ones and those through cell corners) on
the CPU: they obey the limit of steps they are given and say so, and the default
one, 4 (W + H) + 64, is never in their way: also where every node on the way has
to be opened, from each climb limit."""

import ctypes
import os
import subprocess

import numpy as np
import pytest

import synth
from test_cast_cpu import ROOT, S, _levels, _lattice

SHIM = r"""
#include "hf_cast.h"
using namespace hf;
extern "C" void run(const uint32_t *words, const uint32_t *off, const uint32_t *stride,
                    const uint32_t *rows, int levels, const int32_t *rays, long n, int mip,
                    int limit, uint8_t *face, uint32_t *status) {
    LevelDev lv[kMaxLevels + 1];
    for (int k = 0; k <= levels; ++k) lv[k] = LevelDev{words + off[k], stride[k], rows[k]};
    for (long i = 0; i < n; ++i) {
        const int32_t *q = rays + 6 * i;
        const BeamDir d = beam_dir(q[3], q[4], q[5]);
        const Ray r{q[0], q[1], q[2], q[3], q[4], q[5]};
        Hit h;
        Counters c{0, 0};
        cast_general<false, false>(lv, beam_unray(d, beam_ray(d, r), q[2], q[5]),
                                   mip < kBeamLevel ? mip : kBeamLevel, mip, limit, h, c, status);
        face[i] = h.face;
    }
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("lone")
    (d / "shim.cpp").write_text(SHIM)
    so = str(d / "lone.so")
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", os.path.join(ROOT, "include"),
                           "-I", os.path.join(cuda, "include"),
                           "-I", os.path.join(ROOT, "paper_2608_17390_gb300", "csrc"),
                           str(d / "shim.cpp"), "-o", so])
    return ctypes.CDLL(so)


def _faces(lib, lv, rays, mip, limit):
    words = np.concatenate([a.ravel() for a in lv])
    off = np.cumsum([0] + [a.size for a in lv[:-1]]).astype(np.uint32)
    stride = np.array([a.shape[1] for a in lv], np.uint32)
    rows = np.array([a.shape[0] for a in lv], np.uint32)
    rays = np.ascontiguousarray(rays, np.int32)
    face, status = np.empty(len(rays), np.uint8), ctypes.c_uint32()
    lib.run(*[ctypes.c_void_p(a.ctypes.data) for a in (words, off, stride, rows)], len(lv) - 1,
            ctypes.c_void_p(rays.ctypes.data), ctypes.c_long(len(rays)), mip, limit,
            ctypes.c_void_p(face.ctypes.data), ctypes.byref(status))
    assert bool(status.value) == (face == 254).any()
    return face


@pytest.mark.parametrize("W,H", [(1, 1), (64, 64), (37, 129), (300, 2), (4096, 3)])
def test_the_default_limit_is_never_reached(lib, W, H):
    rng = np.random.default_rng(W + H)
    # columns of 120 two cells apart, slabs from 200 on: nodes hold both, rays pass between
    h = np.where((np.add.outer(np.arange(H), np.arange(W)) % 2) == 0, 120, 90)
    cells = synth.pack_cells(h, 200, 210, 1).astype(np.uint32)
    lv = _levels(cells)
    n = 300
    o = np.stack([rng.integers(0, W, n) * S, rng.integers(0, H, n) * S, rng.integers(121 * S, 199 * S, n)], 1)
    d = rng.choice([-1, 1], (n, 3)) * np.array([S, S, 0]) + rng.integers(-3, 4, (n, 1)) * np.array([0, 0, 1])
    rays = np.concatenate([np.concatenate([o, d], 1), _lattice(rng, W, H, 1500)])
    for mip in range(len(lv)):
        assert (_faces(lib, lv, rays, mip, 4 * (W + H) + 64) != 254).all(), mip


def test_a_limit_is_obeyed(lib):
    cells = np.full((50, 50), synth.pack_cells(3, 0, 0, 1), np.uint32)
    rays = np.array([[S, S, 10 * S, S, S, 0], [2 * S, 3 * S, 10 * S, 0, 0, -5]])
    assert list(_faces(lib, _levels(cells), rays, 0, 4)) == [254, 5]
    assert list(_faces(lib, _levels(cells), rays, 0, 60)) == [255, 5]
