"""The traversal in beams (csrc/hf_cast.h) against the general one and the
oracle, on the CPU: the parts of both are host code too, so every form of ray
can be compared without a GPU -- corners, boundaries and grazes on a lattice,
directions from one unit to the limit on either axis, rays across the largest
grids, heights to the top of the range, every start level and climb limit,
and warps of rays from scattered to narrow.  The kernel's loop over a warp
(cast_beams in csrc/hf_trace.cu, beam_next in csrc/hf_beam.h) is written out here lane by lane.
"""

import ctypes
import os
import subprocess

import numpy as np
import pytest

import oracle
import synth

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
S = 65536

SHIM = r"""
#include "hf_cast.h"
#include <algorithm>
using namespace hf;
static long beamed = 0;  // rays that a beam decided
// cast_beams of hf_trace.cu and beam_next of hf_beam.h, with the lanes of a warp in turn
template <bool PAIR>
static void beams(const LevelDev *lv, int top_level_of_world, const Ray *r, int n, int mip, Hit *h) {
    const uint32_t W = lv[0].stride, H = lv[0].rows, *cells = lv[0].base;
    BeamDir d[32];
    BeamRay q[32];
    bool todo[32] = {}, alive[32], alone[32] = {};
    float a[32], b[32];
    for (int k = 0; k < n; ++k) {
        h[k].face = kFaceMiss;
        h[k].layer = 255;
        alone[k] = r[k].dx == 0 && r[k].dy == 0;
        if (alone[k]) continue;
        d[k] = beam_dir(r[k].dx, r[k].dy, r[k].dz);
        q[k] = beam_ray(d[k], r[k]);
        int32_t cx, cy;
        cast_cell(r[k], cx, cy);
        todo[k] = (uint32_t)cx < W && (uint32_t)cy < H;
    }
    const float top = (float)((lv[top_level_of_world].base[0] >> 16) & 0xFF);
    const int base_level = std::min(kBeamLevel, mip), top_level = std::min(kBeamTop, mip);
    for (int lead = 0; lead < n; ++lead) {
        if (!todo[lead]) continue;
        const int key = d[lead].key;
        Beam m;
        m.u0 = q[lead].fu;
        m.v0 = q[lead].fv;
        int32_t u0 = 0x7FFFFFFF;
        for (int k = 0; k < n; ++k) {
            beam_place(q[k], m);
            alive[k] = todo[k] && d[k].key == key &&
                       std::fabs(q[k].pv - d[k].rho * q[k].pu) <= kBeamSpread;
            if (alive[k]) todo[k] = false, u0 = std::min(u0, q[k].fu);
        }
        m.u0 = u0;
        for (int k = 0; k < n; ++k)
            if (alive[k]) {
                beam_place(q[k], m);
                a[k] = q[k].pv - d[k].rho * q[k].pu;
                b[k] = q[k].z0 - d[k].sigma * q[k].pu;
            }
        const int32_t limit = key & 2 ? 0 : (int32_t)(key & 4 ? W : H);
        const BeamGrid g = beam_grid(cells, m, key, W, H);
        int32_t u = m.u0;
        int level = base_level;
        while (u < limit) {
            bool any = false;
            m.a0 = m.r0 = m.b0 = m.s0 = 3e38f;
            m.a1 = m.r1 = m.b1 = m.s1 = -3e38f;
            for (int k = 0; k < n; ++k)
                if (alive[k]) {
                    any = true;
                    m.a0 = std::min(m.a0, a[k]), m.a1 = std::max(m.a1, a[k]);
                    m.r0 = std::min(m.r0, d[k].rho), m.r1 = std::max(m.r1, d[k].rho);
                    m.b0 = std::min(m.b0, b[k]), m.b1 = std::max(m.b1, b[k]);
                    m.s0 = std::min(m.s0, d[k].sigma), m.s1 = std::max(m.s1, d[k].sigma);
                }
            if (!any) break;
            u = beam_skip(m, u, limit, top);
            if (u >= limit) break;
            const int least = beam_least(m, u, base_level, top_level);
            level = std::max(level, least);
            const int32_t j = u >> level;
            uint32_t open = 0;
            uint32_t high;
            for (int i = 0; i < 32; ++i)
                open |= (uint32_t)beam_open<PAIR>(lv, m, level, j + i, key, high) << i;
            if (level > least && open) {
                u = std::max(u, (j + __builtin_ctz(open)) * (1 << level));
                level = least;
                continue;
            }
            const bool found = open != 0;
            while (open) {
                const int i = __builtin_ctz(open), run = beam_run(open, i);
                open &= i + run < 32 ? 0xFFFFFFFFu << (i + run) : 0u;
                const int32_t b0 = std::max(u, (j + i) * (1 << level));
                const int32_t b1 = std::min((j + i + run) * (1 << level), limit);
                for (int k = 0; k < n; ++k) {
                    if (!alive[k] || q[k].fu >= b1) continue;
                    BeamWalk w;
                    BeamHit b;
                    if (!beam_enter(d[k], q[k], m, b0 - m.u0, b1 - m.u0, w)) {
                        alive[k] = false;
                        alone[k] = true;
                    }
                    for (int32_t x = std::max(b0, q[k].fu) - m.u0; alive[k] && x < b1 - m.u0; ++x) {
                        BeamColumn c = {};
                        const int at = beam_step<PAIR>(g, d[k], q[k], m, w, x, c);
                        if (at == kBeamOpen)
                            alive[k] = !beam_settle(g, r[k].oz, r[k].dz, d[k], q[k], m, w, x, c, b);
                        else if (at != kBeamGoing)
                            alive[k] = false, alone[k] = at == kBeamCorner;
                        if (at == kBeamOpen && !alive[k])
                            h[k] = beam_hit(b, r[k].oz, r[k].dz, d[k], q[k]);
                        w.row = c.row;
                        w.zl = c.zl;
                    }
                }
            }
            u = (j + 32) * (1 << level);
            if (!found) level = std::min(level + 2, top_level);
        }
    }
    for (int k = 0; k < n; ++k) {
        Counters c{0, 0};
        beamed += !alone[k];
        if (alone[k]) cast_general<false, PAIR>(lv, r[k], base_level, mip, 1 << 30, h[k], c);
    }
}
template <bool PAIR>
static void go(const LevelDev *lv, int levels, const int32_t *rays, long n, int start, int mip,
               int fast, int32_t *out, double *t) {
    for (long i = 0; i < n; i += 32) {
        const int m = (int)std::min<long>(32, n - i);
        Ray r[32];
        Hit h[32];
        for (int k = 0; k < m; ++k) {
            const int32_t *q = rays + 6 * (i + k);
            r[k] = Ray{q[0], q[1], q[2], q[3], q[4], q[5]};
            Counters c{0, 0};
            if (!fast) cast_general<false, PAIR>(lv, r[k], start, mip, 1 << 30, h[k], c);
        }
        if (fast) beams<PAIR>(lv, levels, r, m, mip, h);
        for (int k = 0; k < m; ++k) {
            const bool hit = h[k].face < kFaceError;
            int32_t *o = out + 4 * (i + k);
            o[0] = hit ? h[k].cx : -1;
            o[1] = hit ? h[k].cy : -1;
            o[2] = h[k].layer;
            o[3] = h[k].face;
            t[i + k] = hit ? (double)h[k].tnum / h[k].tden : -1.0;
        }
    }
}
extern "C" long count() { return beamed; }
extern "C" void cast(const uint32_t *words, const uint32_t *off, const uint32_t *stride,
                     const uint32_t *rows, int levels, int pair, const int32_t *rays, long n,
                     int start, int mip, int fast, int32_t *out, double *t) {
    LevelDev lv[kMaxLevels + 1];
    for (int k = 0; k <= levels; ++k) lv[k] = LevelDev{words + off[k], stride[k], rows[k]};
    (pair ? go<true> : go<false>)(lv, levels, rays, n, start, mip, fast, out, t);
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("cast")
    (d / "shim.cpp").write_text(SHIM)
    so = str(d / "cast.so")
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-ffp-contract=off",
                           "-I", os.path.join(ROOT, "include"), "-I", os.path.join(cuda, "include"),
                           "-I", os.path.join(ROOT, "paper_2608_17390_gb300", "csrc"),
                           str(d / "shim.cpp"), "-o", so])
    return ctypes.CDLL(so)


def _levels(cells):
    """Node-form words of every level, and the cells as the kernels store them."""
    h0, h1, h2, mat = (a.astype(np.uint32) for a in synth.unpack_cells(cells))
    slab = h1 > h0
    lv = [np.stack([h0, np.where(slab, h1, 255), np.where(slab, h2, h0)])]
    while max(lv[-1].shape[1:]) > 1:
        a = lv[-1]
        H, W = a.shape[1:]
        p = np.zeros((3, (H + 1) & ~1, (W + 1) & ~1), np.uint32)
        p[1] = 255
        p[:, :H, :W] = a
        q = p.reshape(3, p.shape[1] // 2, 2, p.shape[2] // 2, 2)
        lv.append(np.stack([q[0].max((1, 3)), q[1].min((1, 3)), q[2].max((1, 3))]))
    words = [a[0] | (a[1] << 8) | (a[2] << 16) for a in lv]
    words[0] = words[0] | (mat << 24)
    return [np.ascontiguousarray(w, np.uint32) for w in words]


class World:
    def __init__(self, lib, cells, texels=None):
        self.lib, self.cells, self.pair = lib, cells, texels is not None
        words = _levels(cells)
        flat = [w.ravel() for w in words]
        if self.pair:
            flat[0] = np.ascontiguousarray(texels).view(np.uint32).ravel()
        self.words = np.concatenate(flat)
        self.off = np.cumsum([0] + [f.size for f in flat[:-1]]).astype(np.uint32)
        self.stride = np.array([w.shape[1] for w in words], np.uint32)
        self.rows = np.array([w.shape[0] for w in words], np.uint32)
        self.L = len(words) - 1

    def cast(self, rays, start, mip, fast):
        rays = np.ascontiguousarray(rays, np.int32)
        n = len(rays)
        out, t = np.empty((n, 4), np.int32), np.empty(n)
        p = [ctypes.c_void_p(a.ctypes.data) for a in
             (self.words, self.off, self.stride, self.rows)]
        self.lib.cast(*p, self.L, int(self.pair), ctypes.c_void_p(rays.ctypes.data),
                      ctypes.c_long(n), int(start), int(mip), int(fast),
                      ctypes.c_void_p(out.ctypes.data), ctypes.c_void_p(t.ctypes.data))
        return out, t

    def check(self, rays, mips=None):
        want, wt = self.cast(rays, 0, 0, False)
        for mip in (range(self.L + 1) if mips is None else mips):
            for start in {0, mip // 2, mip}:
                for fast in (False, True):
                    got, gt = self.cast(rays, start, mip, fast)
                    bad = np.nonzero((got != want).any(1) | (gt != wt))[0]
                    assert bad.size == 0, "%d rays differ (start %d, mip %d, fast %d): %s got %s want %s" % (
                        bad.size, start, mip, fast, rays[bad[0]], got[bad[0]], want[bad[0]])
        return want


def _lattice(rng, W, H, n):
    """Rays through exact corners, boundaries, tops and undersides."""
    q = rng.choice([S // 2, S, S // 4, 2 * S, 1], n)
    o = np.stack([rng.integers(0, W * S, n) // q * q, rng.integers(0, H * S, n) // q * q,
                  rng.integers(0, 300, n) * S + rng.choice([0, 0, 1, S // 2], n)], 1)
    d = rng.integers(-4, 5, (n, 3)) * rng.choice([1, 7, 1000, S, 300000], n)[:, None]
    return np.concatenate([o, d], 1)


def _spread(rng, W, H, n, zmax=400):
    """Directions from one unit to the limit, independently on each axis."""
    o = np.stack([rng.integers(0, W * S, n), rng.integers(0, H * S, n),
                  rng.integers(0, zmax * S, n)], 1)
    mag = np.minimum(2.0 ** rng.uniform(0, 21, (n, 3)), 2**21 - 1).astype(np.int64)
    d = mag * rng.choice([-1, 1], (n, 3))
    d[: n // 4, 2] = -np.maximum(1, np.abs(d[: n // 4, :2]).max(1) // rng.integers(1, 60, n // 4))
    return np.concatenate([o, d], 1)


@pytest.mark.parametrize("W,H,slab,walls", [(1, 1, 0.0, 0), (5, 3, 0.5, 1), (64, 64, 0.4, 8),
                                            (37, 129, 0.3, 6), (300, 17, 0.0, 4)])
def test_beams_equal_general_at_every_level(lib, W, H, slab, walls):
    rng = np.random.default_rng(W * 1000 + H)
    cells, _ = synth.make_grid(W, H, seed=W + H, slab_frac=slab, n_walls=walls)
    w = World(lib, cells)
    rays = np.concatenate([_lattice(rng, W, H, 6000), _spread(rng, W, H, 6000)])
    got = w.check(rays)
    o = oracle.trace_rays(cells, rays[:, :3], rays[:, 3:])
    hit = o["hit_cell"] != 0xFFFFFFFF
    cell = np.where(got[:, 0] < 0, 0xFFFFFFFF, got[:, 1].astype(np.int64) * W + got[:, 0])
    assert (cell == o["hit_cell"]).all() and (got[:, 3] == o["face"]).all()
    assert (got[hit, 2] == o["layer"][hit]).all()


def test_extreme_heights_and_wide_grids(lib):
    """Origins to the top of the range, and grids as wide and tall as can be."""
    for W, H in ((16384, 3), (2, 16384), (2048, 700)):
        rng = np.random.default_rng(W)
        cells, _ = synth.make_grid(W, H, seed=9, slab_frac=0.3, n_walls=20)
        w = World(lib, cells)
        rays = np.concatenate([_spread(rng, W, H, 3000, 4096), _spread(rng, W, H, 3000),
                               _lattice(rng, W, H, 2000)])
        # long level rays: along the grid, just above and under the solids
        n = 2000
        o = np.stack([rng.integers(0, W * S, n), rng.integers(0, H * S, n),
                      rng.integers(60 * S, 260 * S, n)], 1)
        d = np.stack([rng.integers(-H, H, n) if W < H else rng.integers(2**18, 2**20, n),
                      rng.integers(2**18, 2**20, n) if W < H else rng.integers(-H, H, n),
                      rng.integers(-900, 900, n)], 1)
        w.check(np.concatenate([rays, np.concatenate([o, d], 1)]), mips=(0, 3, 6, 10, w.L))


def test_bundles(lib):
    """Warps of rays that stay together: from one point into a narrow cone, and
    from neighbouring points along one direction (what pixels and their
    shadow rays are), over caves and walls."""
    rng = np.random.default_rng(4)
    W, H = 700, 900
    w = World(lib, synth.make_grid(W, H, seed=12, slab_frac=0.4, n_walls=300)[0])
    rays = []
    for g in range(600):
        o = np.array([rng.integers(0, W * S), rng.integers(0, H * S), rng.integers(20 * S, 400 * S)])
        d = rng.integers(-2**20, 2**20, 3)
        d[2] //= rng.choice([1, 3, 40])
        if g % 3 == 0:
            d[rng.integers(2)] //= rng.choice([1, 1000, 2**20])
        spread = rng.choice([300, 3000, 60000])
        if g % 2:
            ray = np.concatenate([np.tile(o, (32, 1)), d + rng.integers(-spread, spread, (32, 3))], 1)
        else:
            far = rng.choice([S // 4, 4 * S, 60 * S])
            p = o + rng.integers(-far, far, (32, 3))
            p = np.clip(p, 0, [W * S - 1, H * S - 1, 400 * S])
            ray = np.concatenate([p, np.tile(d, (32, 1))], 1)
        ray[:, 3:] = np.clip(ray[:, 3:], -2**21 + 1, 2**21 - 1)
        rays.append(ray)
    got = w.check(np.concatenate(rays), mips=(0, 1, 4, w.L))
    assert 0.2 < (got[:, 0] >= 0).mean() < 0.95


def test_paired_texels(lib):
    rng = np.random.default_rng(8)
    cells = synth.pairify(synth.make_grid(130, 77, seed=5, slab_frac=0.4, n_walls=5)[0])
    w = World(lib, cells, synth.encode_pairs(cells))
    want = World(lib, cells)
    rays = np.concatenate([_lattice(rng, 130, 77, 4000), _spread(rng, 130, 77, 4000)])
    assert (w.check(rays, mips=(0, 4, w.L)) == want.check(rays, mips=(3,))).all()
