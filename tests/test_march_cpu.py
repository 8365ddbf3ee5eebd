"""The march in beams (csrc/hf_march.h, hf_cast.h) against every sample, on the
CPU, where a sample's rounding shows: starts 1 to 32 units either side of cell
and 32-cell boundaries at coordinates up to 16384, steep rays both ways on both
axes beside high columns, under slabs, and views from straight down to level.
A hit has to be the one of the marcher's oracle bit for bit.  The kernel's loop
over a warp (march_beams in csrc/hf_march.cu, beam_next in csrc/hf_beam.h) is
written out here lane by lane.
"""

import ctypes
import os
import subprocess

import numpy as np
import pytest

import synth
from oracle import march
from test_cast_cpu import ROOT, S, _levels

SHIM = r"""
#include "hf_march.h"
#include <algorithm>
using namespace hf;
struct World {
    LevelDev lv[kMaxLevels + 1];
    int top;
};
static bool solid(const World &w, const MarchSpot &s, bool &floor_) {
    return (uint32_t)s.cx < w.lv[0].stride && (uint32_t)s.cy < w.lv[0].rows &&
           march_solid(w.lv[0].base[(uint32_t)s.cy * w.lv[0].stride + s.cx], s.z, floor_);
}
static int32_t samples(const World &w, const MarchRay &m, int32_t i, int32_t last) {
    bool f;
    for (; i <= last; ++i)
        if (solid(w, march_spot(m, rn_mul((float)i, m.dt)), f)) return i;
    return 0;
}
static void march_warp(const World &w, const Ray *r, const MarchRay *m, int n, int32_t steps,
                       int32_t *found) {
    BeamDir d[32];
    BeamRay q[32];
    MarchRate rate[32];
    bool todo[32], alive[32];
    float a[32], b[32];
    int32_t next[32];
    for (int k = 0; k < n; ++k) {
        found[k] = 0;
        d[k] = beam_dir(r[k].dx, r[k].dy, r[k].dz);
        q[k] = beam_ray(d[k], r[k]);
        rate[k] = march_rate(m[k], d[k]);
        todo[k] = d[k].du != 0 && m[k].dt > 1e-9f && m[k].dt < 1e9f;
        if (!todo[k]) found[k] = samples(w, m[k], 1, steps);
    }
    const uint32_t W = w.lv[0].stride, H = w.lv[0].rows;
    const float top = (float)((w.lv[w.top].base[0] >> 16) & 0xFF);
    const int base_level = std::min(kBeamLevel, w.top), top_level = std::min(kBeamTop, w.top);
    for (int lead = 0; lead < n; ++lead) {
        if (!todo[lead]) continue;
        const int key = d[lead].key;
        Beam bm;
        bm.u0 = q[lead].fu;
        bm.v0 = q[lead].fv;
        for (int k = 0; k < n; ++k) {
            alive[k] = todo[k] && d[k].key == key;
            if (!alive[k]) continue;
            todo[k] = false;
            beam_place(q[k], bm);
            a[k] = q[k].pv - d[k].rho * q[k].pu;
            b[k] = q[k].z0 - d[k].sigma * q[k].pu;
            next[k] = 1;
        }
        const int32_t limit = key & 2 ? 0 : (int32_t)(key & 4 ? W : H);
        int32_t u = bm.u0 - 1;
        int level = base_level;
        while (u < limit) {
            bool any = false;
            bm.a0 = bm.r0 = bm.b0 = bm.s0 = 3e38f;
            bm.a1 = bm.r1 = bm.b1 = bm.s1 = -3e38f;
            for (int k = 0; k < n; ++k)
                if (alive[k]) {
                    any = true;
                    bm.a0 = std::min(bm.a0, a[k]), bm.a1 = std::max(bm.a1, a[k]);
                    bm.r0 = std::min(bm.r0, d[k].rho), bm.r1 = std::max(bm.r1, d[k].rho);
                    bm.b0 = std::min(bm.b0, b[k]), bm.b1 = std::max(bm.b1, b[k]);
                    bm.s0 = std::min(bm.s0, d[k].sigma), bm.s1 = std::max(bm.s1, d[k].sigma);
                }
            if (!any) break;
            u = beam_skip<true>(bm, u, limit, top);
            if (u >= limit) break;
            const int least = beam_least(bm, u, base_level, top_level);
            level = std::max(level, least);
            const int32_t j = u >> level;
            uint32_t open = 0, high[32];
            for (int i = 0; i < 32; ++i)
                open |= (uint32_t)beam_open<false, true>(w.lv, bm, level, j + i, key, high[i]) << i;
            if (level > least && open) {
                u = std::max(u, (j + __builtin_ctz(open)) * (1 << level));
                level = least;
                continue;
            }
            const bool met = open != 0;
            open = beam_joined(open);
            while (open) {
                const int i = __builtin_ctz(open), run = beam_run(open, i);
                open &= i + run < 32 ? 0xFFFFFFFFu << (i + run) : 0u;
                const int32_t b0 = std::max(u, (j + i) * (1 << level));
                const int32_t b1 = std::min((j + i + run) * (1 << level), limit);
                uint32_t peak = 0;
                for (int t = i; t < i + run; ++t) peak = std::max(peak, high[t]);
                for (int k = 0; k < n; ++k) {
                    if (!alive[k]) continue;
                    const MarchRun mr = march_run(m[k], rate[k], q[k].pu, (float)(b0 - bm.u0),
                                                  (float)(b1 - bm.u0), (float)peak, (float)steps);
                    alive[k] = !mr.past;
                    const int32_t at =
                        alive[k] ? samples(w, m[k], std::max(next[k], mr.first), mr.last) : 0;
                    if (at && march_column(march_spot(m[k], rn_mul((float)at, m[k].dt)), key) < b1)
                        found[k] = at;
                    next[k] = std::max(next[k], mr.done);
                    alive[k] = alive[k] && !found[k];
                }
            }
            u = (j + 32) * (1 << level);
            if (!met) level = std::min(level + 2, top_level);
        }
    }
}
// found: the first solid sample, in beams (fast) or of all; hit: the hit that four
// bisections leave
extern "C" void run(const uint32_t *words, const uint32_t *off, const uint32_t *stride,
                    const uint32_t *rows, int levels, const int32_t *rays, long n, int32_t steps,
                    float far_dist, int fast, int32_t *found, uint32_t *cell, uint8_t *layer,
                    float *depth) {
    World w;
    w.top = levels;
    for (int k = 0; k <= levels; ++k) w.lv[k] = LevelDev{words + off[k], stride[k], rows[k]};
    for (long i = 0; i < n; i += 32) {
        const int c = (int)std::min<long>(32, n - i);
        Ray r[32];
        MarchRay m[32];
        float len[32];
        for (int k = 0; k < c; ++k) {
            const int32_t *p = rays + 6 * (i + k);
            r[k] = Ray{p[0], p[1], p[2], p[3], p[4], p[5]};
            float f[6];
            for (int t = 0; t < 6; ++t) f[t] = (float)p[t] * (1.0f / 65536.0f);
            m[k] = MarchRay{f[0], f[1], f[2], f[3], f[4], f[5], 0.0f};
            len[k] = sqrtf(f[3] * f[3] + f[4] * f[4] + f[5] * f[5]);
            float t_end = far_dist / len[k];
            if (f[5] < 0.0f && -f[2] / f[5] < t_end) t_end = -f[2] / f[5];
            m[k].dt = t_end / (float)(steps + 1);
        }
        if (fast) march_warp(w, r, m, c, steps, found + i);
        for (int k = 0; k < c; ++k) {
            if (!fast) found[i + k] = samples(w, m[k], 1, steps);
            cell[i + k] = 0xFFFFFFFFu;
            layer[i + k] = 255;
            depth[i + k] = INFINITY;
            if (!found[i + k]) continue;
            float ta = (float)(found[i + k] - 1) * m[k].dt, tb = (float)found[i + k] * m[k].dt;
            bool fl;
            for (int t = 0; t < 4; ++t) {
                const float tm = (ta + tb) * 0.5f;
                if (solid(w, march_spot(m[k], tm), fl)) tb = tm;
                else ta = tm;
            }
            const MarchSpot s = march_spot(m[k], tb);
            solid(w, s, fl);
            cell[i + k] = (uint32_t)s.cy * w.lv[0].stride + s.cx;
            layer[i + k] = fl ? 0 : 1;
            depth[i + k] = tb * len[k];
        }
    }
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("march")
    (d / "shim.cpp").write_text(SHIM)
    so = str(d / "march.so")
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-ffp-contract=off",
                           "-I", os.path.join(ROOT, "include"), "-I", os.path.join(cuda, "include"),
                           "-I", os.path.join(ROOT, "paper_2608_17390_gb300", "csrc"),
                           str(d / "shim.cpp"), "-o", so])
    return ctypes.CDLL(so)


class World:
    def __init__(self, lib, cells):
        self.lib, self.cells = lib, cells
        lv = _levels(cells)
        self.words = np.concatenate([a.ravel() for a in lv])
        self.off = np.cumsum([0] + [a.size for a in lv[:-1]]).astype(np.uint32)
        self.stride = np.array([a.shape[1] for a in lv], np.uint32)
        self.rows = np.array([a.shape[0] for a in lv], np.uint32)

    def march(self, rays, steps, far, fast):
        n = len(rays)
        out = dict(found=np.empty(n, np.int32), hit_cell=np.empty(n, np.uint32),
                   layer=np.empty(n, np.uint8), depth=np.empty(n, np.float32))
        p = [ctypes.c_void_p(a.ctypes.data) for a in (self.words, self.off, self.stride, self.rows)]
        self.lib.run(*p, len(self.off) - 1, ctypes.c_void_p(rays.ctypes.data), ctypes.c_long(n),
                     int(steps), ctypes.c_float(far), int(fast),
                     *[ctypes.c_void_p(a.ctypes.data) for a in out.values()])
        return out

    def check(self, rays, steps=128, far=600.0, every=1):
        """Beams equal every sample; each `every`-th ray's hit equals the oracle's."""
        rays = np.ascontiguousarray(rays, np.int32)
        want, got = self.march(rays, steps, far, False), self.march(rays, steps, far, True)
        bad = np.nonzero(got["found"] != want["found"])[0]
        assert bad.size == 0, "%d rays differ: %s sample %d, first solid %d" % (
            bad.size, rays[bad[0]].tolist(), got["found"][bad[0]], want["found"][bad[0]])
        few = rays[::every]
        ref = march.march(self.cells, few[:, :3], few[:, 3:], steps=steps, far=far)
        for k in ("hit_cell", "layer"):
            assert np.array_equal(got[k][::every], ref[k]), k
        assert np.array_equal(got["depth"][::every].view(np.uint32), ref["depth"].view(np.uint32))
        return got


def _world(lib, W, H, seed, high):
    """Floors of 10 to 40 with columns up to `high`, a third of them slabs."""
    rng = np.random.default_rng(seed)
    h0 = rng.integers(10, 41, (H, W)).astype(np.uint32)
    wall = rng.random((H, W)) < 0.1
    h0 = np.where(wall, rng.integers(60, high + 1, (H, W)), h0).astype(np.uint32)
    slab = rng.random((H, W)) < 0.3
    h1 = np.where(slab, np.minimum(h0 + 20, 254), 0)
    return World(lib, synth.pack_cells(h0, h1, np.where(slab, np.minimum(h1 + 9, 255), 0), 1)
                 .astype(np.uint32))


def test_a_view_straight_down_beside_a_high_column(lib):
    """A camera four units short of the column: its rounded origin lies over it."""
    cells = np.full((24, 16384), synth.pack_cells(10, 0, 0, 1), np.uint32)
    cells[:, 9568] = synth.pack_cells(200, 0, 0, 1)
    w = World(lib, cells)
    for units in (1, 4, 16):
        o = [9568 * S - units, 12 * S, 100 * S]
        d = np.array([[a, b, -524288] for a in range(-1570, 1571, 628) for b in range(-1570, 1571, 628)]
                     + [[-314, 314, -524288]])
        got = w.check(np.concatenate([np.tile(o, (len(d), 1)), d], 1))
        assert (got["found"] == 1).any()


@pytest.mark.parametrize("wide", [True, False])
@pytest.mark.parametrize("steps,far", [(128, 600.0), (1000, 600.0), (33, 5000.0)])
def test_starts_beside_boundaries(lib, wide, steps, far):
    W, H = (16384, 24) if wide else (24, 16384)
    w = _world(lib, W, H, steps, 230)
    rng = np.random.default_rng(steps + wide)
    n = 3000  # warps
    at = np.minimum(2.0 ** rng.uniform(8, 14, n), 16383).astype(np.int64)
    at = np.where(rng.random(n) < 0.3, at & ~31, at)
    side = rng.choice([-1, 1], n) * rng.integers(1, 33, n)
    along = np.clip(at * S + side, 0, 16384 * S - 1)
    across = rng.integers(1, 23, n) * S + rng.choice([0, 1, -1, 30000], n)
    z = rng.integers(0, 300 * S, n)
    o = np.stack([along, across, z] if wide else [across, along, z], 1)
    steep = (2.0 ** rng.uniform(0, 14, (n, 1, 1))).astype(np.int64)
    d = np.empty((n, 32, 3), np.int64)
    d[..., :2] = np.round(rng.uniform(-1, 1, (n, 32, 2)) * steep)
    d[..., 2] = np.where(rng.random(n) < 0.75, -524288, 524288)[:, None]
    w.check(np.concatenate([np.repeat(o[:, None], 32, 1), d], 2).reshape(-1, 6), steps, far, every=97)


def test_warps_of_a_view(lib):
    """8 x 4 pixels of views in all directions, from the air, under slabs and inside."""
    W, H = 700, 5000
    w = _world(lib, W, H, 3, 120)
    rng = np.random.default_rng(5)
    n = 1500
    o = np.stack([rng.integers(0, W * S, n), rng.integers(0, H * S, n), rng.integers(0, 400 * S, n)], 1)
    o[::4, :2] = o[::4, :2] // S * S
    mid = rng.integers(-2**20, 2**20, (n, 1, 3)) // rng.choice([1, 1, 50], (n, 1, 3))
    px = rng.integers(200, 3000, (n, 1, 1))
    k = np.arange(32)
    d = mid + px * np.stack([k % 8, k // 8, (k % 8) - (k // 8)], 1)[None]
    d[..., 2] -= 1
    w.check(np.concatenate([np.repeat(o[:, None], 32, 1), d], 2).reshape(-1, 6), 128, 600.0, every=31)
    w.check(np.concatenate([np.repeat(o[:, None], 32, 1), d], 2).reshape(-1, 6), 700, 90.0, every=311)


def test_every_key_and_a_one_cell_world(lib):
    w = World(lib, np.full((1, 1), synth.pack_cells(9, 40, 60, 2), np.uint32))
    rng = np.random.default_rng(1)
    o = rng.integers(0, S, (64, 1, 3)) + np.array([0, 0, 20 * S])
    d = rng.integers(-3, 4, (64, 32, 3)) * rng.choice([1, 1000, 300000], (64, 1, 1))
    d[(d == 0).all(2)] = (0, 0, -5)
    w.check(np.concatenate([np.repeat(o, 32, 1), d], 2).reshape(-1, 6), 128, 600.0)


def test_a_higher_column_right_after_a_run(lib):
    """Samples so dense that several lie in the 0.02 columns past a run of low
    columns, at whose end a wall stands that the first of them is in already."""
    h = np.full((8, 300), 50)
    h[:, 162:] = 200  # where 32 stretches of two columns end
    w = World(lib, synth.pack_cells(h, 0, 0, 1).astype(np.uint32))
    rays = [[100 * S + S // 2, 4 * S, int((z + 2 * 61.5) * S), S, 0, -2 * S]
            for z in np.linspace(50.0, 50.04, 81)]
    got = w.check(np.array(rays), 65000, 150.0)
    assert (got["hit_cell"] % 300 == 162).sum() > 30
