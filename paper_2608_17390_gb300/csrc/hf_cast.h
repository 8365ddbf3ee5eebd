// hf_cast.h -- the traversal of rays through the cells and their pyramid.
//
// Two traversals give the same hit:
//
//   cast_single   one ray, hierarchical DDA, every decision on rationals
//                 num/den with 64-bit products (hf_single.cu).  Counts fetches,
//                 obeys a step limit of the caller's.
//   beam_*        the parts of a warp's traversal (hf_trace.cu): the rays of a
//                 warp that go the same way are bounded by one beam, whose 32
//                 next stretches are tested by the 32 lanes at once; rays are
//                 walked, column by column in float with error bounds, only
//                 through stretches that the beam does not prove empty.  What
//                 the bounds leave open is decided exactly, on rationals, and
//                 a ray through a cell corner is left to the other (cast_general).
//
// The functions are host code too, so that the two can be compared on a CPU.
#pragma once

#include <cmath>
#include <cstdint>
#include <cstdlib>
#include <cstring>

#include "hf_internal.h"

#ifdef __CUDACC__
#define HF_HD __host__ __device__ __forceinline__
#else
#define HF_HD inline
#endif

namespace hf {

struct Ray {
    int32_t ox, oy, oz, dx, dy, dz;
};

// The ray of a camera's pixel.
HF_HD Ray primary_ray(const CamDev &c, int32_t px, int32_t py) {
    const int32_t a = 2 * px + 1 - (int32_t)c.w;
    const int32_t b = (int32_t)c.h - 1 - 2 * py;
    return Ray{c.o[0], c.o[1], c.o[2], c.F[0] + a * c.R[0] + b * c.U[0],
               c.F[1] + a * c.R[1] + b * c.U[1], c.F[2] + a * c.R[2] + b * c.U[2]};
}

// One pyramid level as the traversal reads it (a per-block shared table, so
// lanes at different levels read it in one shared-memory access).
struct LevelDev {
    const uint32_t *base;
    uint32_t stride, rows;
};

struct Hit {
    int32_t cx, cy;
    int32_t tnum, tden;  // hit time tnum / tden
    uint32_t word;       // hit cell word
    uint8_t layer, face;
};

struct Counters {
    uint32_t nodes, cells;
};

HF_HD uint32_t cast_load(const uint32_t *p) {
#ifdef __CUDA_ARCH__
    return __ldg(p);
#else
    return *p;
#endif
}

HF_HD float cast_rcp(float v) {
#ifdef __CUDA_ARCH__
    return __frcp_rn(v);
#else
    return 1.0f / v;
#endif
}

// 1 / v to a relative 2^-22.
HF_HD float cast_rcp_fast(float v) {
#ifdef __CUDA_ARCH__
    return __fdividef(1.0f, v);
#else
    return 1.0f / v;
#endif
}

// Maximum of each 16-bit half.
HF_HD uint32_t max_halves(uint32_t a, uint32_t b) {
#ifdef __CUDA_ARCH__
    return __vmaxu2(a, b);
#else
    const uint32_t al = a & 0xFFFF, bl = b & 0xFFFF, ah = a >> 16, bh = b >> 16;
    return (al > bl ? al : bl) | (ah > bh ? ah : bh) << 16;
#endif
}

HF_HD int32_t float_bits(float v) {
#ifdef __CUDA_ARCH__
    return __float_as_int(v);
#else
    int32_t i;
    memcpy(&i, &v, sizeof i);
    return i;
#endif
}

// Bit 0 of a status word (none: no word): a ray was given up.
HF_HD void cast_failed(uint32_t *status) {
    if (!status) return;
#ifdef __CUDA_ARCH__
    atomicOr(status, 1u);
#else
    *status |= 1;
#endif
}

// sign carrier of z(t) - h S for t = num / den (den > 0):  (oz - hS) den + num dz
HF_HD int64_t zd(int32_t oz_minus_hs, int32_t dz, int32_t num, int32_t den) {
    return (int64_t)oz_minus_hs * den + (int64_t)num * dz;
}

// Node-form word of node (x, y) of the level `lv` for the storage the kernel
// was instantiated for (the choice is made at compile time; `level` matters
// for paired texels only).
template <bool PAIR>
HF_HD uint32_t cast_word(const LevelDev &lv, int level, int32_t x, int32_t y) {
    if (PAIR && level == 0)
        return pair_node(cast_load(lv.base + (uint32_t)y * (lv.stride >> 1) + ((uint32_t)x >> 1)),
                         (uint32_t)x & 1);
    return cast_load(lv.base + (uint32_t)y * lv.stride + (uint32_t)x);
}

// The two-interval test of one cell over [tin, tout] (tout finite).
// Returns true and fills h on a hit; false exactly when nothing is solid
// along the segment.
HF_HD bool leaf_test(int32_t oz, int32_t dz, uint32_t word, int32_t tin_num, int32_t tin_den,
                     int32_t tout_num, int32_t tout_den, uint8_t entry_face, Hit &h) {
    const int32_t h0 = word & 0xFF, h1 = (word >> 8) & 0xFF, h2 = (word >> 16) & 0xFF;
    const bool slab = h2 > h0;  // level-0 words are in node form
    const int32_t a0 = oz - (h0 << kShift);
    const int64_t zin0 = zd(a0, dz, tin_num, tin_den);
    if (zin0 <= 0) {
        h.layer = 0;
        h.face = entry_face;
        h.tnum = tin_num;
        h.tden = tin_den;
        return true;
    }
    const int32_t a1 = oz - (h1 << kShift), a2 = oz - (h2 << kShift);
    int64_t zin1 = 0, zin2 = 0;
    if (slab) {
        zin1 = zd(a1, dz, tin_num, tin_den);
        zin2 = zd(a2, dz, tin_num, tin_den);
        if (zin1 >= 0 && zin2 <= 0) {
            h.layer = 1;
            h.face = entry_face;
            h.tnum = tin_num;
            h.tden = tin_den;
            return true;
        }
    }
    if (dz < 0) {
        if (slab && zin2 > 0 && zd(a2, dz, tout_num, tout_den) <= 0) {
            h.layer = 1;
            h.face = kFacePZ;
            h.tnum = a2;
            h.tden = -dz;
            return true;
        }
        if (zd(a0, dz, tout_num, tout_den) <= 0) {
            h.layer = 0;
            h.face = kFacePZ;
            h.tnum = a0;
            h.tden = -dz;
            return true;
        }
    } else if (dz > 0) {
        if (slab && zin1 < 0 && zd(a1, dz, tout_num, tout_den) >= 0) {
            h.layer = 1;
            h.face = kFaceNZ;
            h.tnum = -a1;
            h.tden = dz;
            return true;
        }
    }
    return false;
}

// A vertical ray (dx = dy = 0) stays in its start column for all t >= 0.
// Writes h only when the ray hits.
HF_HD bool vertical_test(const Ray &r, uint32_t word, Hit &h) {
    const int32_t h0 = word & 0xFF, h1 = (word >> 8) & 0xFF, h2 = (word >> 16) & 0xFF;
    const bool slab = h2 > h0;  // level-0 words are in node form
    const int32_t a0 = r.oz - (h0 << kShift), a1 = r.oz - (h1 << kShift),
                  a2 = r.oz - (h2 << kShift);
    uint8_t layer, face;
    int32_t tnum = 0, tden = 1;
    if (a0 <= 0) {
        layer = 0;
        face = kFaceInside;
    } else if (slab && a1 >= 0 && a2 <= 0) {
        layer = 1;
        face = kFaceInside;
    } else if (r.dz < 0) {
        face = kFacePZ;
        tden = -r.dz;
        layer = (slab && a2 > 0) ? 1 : 0;
        tnum = layer ? a2 : a0;
    } else if (r.dz > 0 && slab && a1 < 0) {
        layer = 1;
        face = kFaceNZ;
        tnum = -a1;
        tden = r.dz;
    } else {
        return false;
    }
    h.layer = layer;
    h.face = face;
    h.tnum = tnum;
    h.tden = tden;
    return true;
}

// The cell a ray occupies just after t = 0.
HF_HD void cast_cell(const Ray &r, int32_t &cx, int32_t &cy) {
    cx = (r.ox >> kShift) - (r.dx < 0 && (r.ox & 0xFFFF) == 0 ? 1 : 0);
    cy = (r.oy >> kShift) - (r.dy < 0 && (r.oy & 0xFFFF) == 0 ? 1 : 0);
}

// Exact first hit of one ray.  h.face = kFaceMiss on a miss, kFaceError when
// max_steps iterations did not finish the ray, which status is told too (where it
// happens: told by h.face afterwards, it cost the kernels of beams up to 1 %, told
// from two places 6 %, by their registers).  lvt: the world's levels; W, H and
// cells are those of level 0.
//
// State: the node (nx, ny) at `level` that holds the ray just after t_in.
// Skipping an empty node changes only the node index on the exit axis; the
// finer bits on the other axis are found when the traversal descends, by
// asking whether the ray has crossed the child midline by t_in (exact
// cross-multiplied time comparison).  Every interior cell boundary of a node
// is the midline of exactly one sub-level, so a ray that enters a cell through
// its Y side while also crossing an X cell boundary (a corner) is detected on
// the way down and reported with the X face (X_TIME: and with the time as that
// boundary's, over |dx|).
// EMPTY_FIRST picks the order of the two outcomes of the node test in the
// code (empty: advance; else descend or hit); which order runs faster depends
// on the kernel (measured: empty first with shadow rays, the other without).
template <bool STATS, bool PAIR, bool EMPTY_FIRST, bool X_TIME>
HF_HD void cast_single(int32_t W, int32_t H, const uint32_t *cells, const LevelDev *lvt,
                       const Ray &r, int start_level, int mip_start, int max_steps,
                       uint32_t *status, Hit &h, Counters &cnt) {
    h.face = kFaceMiss;
    h.layer = 255;
    // (abs, and not a choice of sign: the compiler then knows that both are
    // positive; the products below cost 5 % of the kernel's time otherwise)
    const int32_t adx = abs(r.dx), ady = abs(r.dy);
    int32_t cx, cy;
    cast_cell(r, cx, cy);
    if ((uint32_t)cx >= (uint32_t)W || (uint32_t)cy >= (uint32_t)H) return;

    if (adx == 0 && ady == 0) {
        const uint32_t word = cast_word<PAIR>(LevelDev{cells, (uint32_t)W, (uint32_t)H}, 0, cx, cy);
        if (STATS) cnt.cells++;
        if (vertical_test(r, word, h)) {
            h.cx = cx;
            h.cy = cy;
            h.word = word;
        }
        return;
    }

    // Per-ray sign constants.  A zero direction component counts as positive:
    // its exit distance is then positive and never the smaller one, so the
    // ray never leaves through that axis.
    const int32_t gx = r.dx < 0 ? -1 : 1, gy = r.dy < 0 ? -1 : 1;  // step per exit
    const int32_t px = r.dx < 0 ? 0 : 1, py = r.dy < 0 ? 0 : 1;    // exit side offset
    const int32_t qx = px ^ 1, qy = py ^ 1;
    const int32_t kx = -gx * r.ox, ky = -gy * r.oy;
    const uint8_t face_x = r.dx < 0 ? kFacePX : kFaceNX;  // entry face of an x crossing
    const uint8_t face_y = r.dy < 0 ? kFacePY : kFaceNY;
    int level = start_level;  // <= mip_start, the coarsest level the ray climbs to
    int32_t nx = cx >> level, ny = cy >> level;
    int32_t tin_num = 0, tin_den = 1;
    uint8_t entry = kFaceInside;

    for (int it = 0;; ++it) {
        // one bounds check per iteration, after every advance, ascent or
        // descent: an index past the level's end, or below 0, means the ray
        // has left the grid.  An ascent keeps the crossed axis out of range
        // (it follows a step onto an even index n >= ceil(E / 2^l), so
        // n / 2 >= ceil(E / 2^(l+1)); or onto -1, and -1 >> 1 = -1).  At an
        // exact corner the other axis may come back in range, in a partial
        // node past the grid's edge; the ray only moves further out, and a
        // descent there lands on an out-of-range child, so it still misses.
        // A ray that leaves on its last allowed iteration is a miss, not a
        // step-limit error.
        const LevelDev lv = lvt[level];
        if ((uint32_t)nx >= lv.stride || (uint32_t)ny >= lv.rows) return;
        if (it == max_steps) break;
        const int32_t bx = (nx + px) * (1 << level);  // exit boundary (cells)
        const int32_t by = (ny + py) * (1 << level);
        const int32_t numx = gx * (bx * (1 << kShift)) + kx;  // > 0
        const int32_t numy = gy * (by * (1 << kShift)) + ky;
        const int64_t cmp = (int64_t)numx * ady - (int64_t)numy * adx;  // < 0: x exits first
        const bool xfirst = cmp <= 0;
        const int32_t tout_num = xfirst ? numx : numy;
        const int32_t tout_den = xfirst ? adx : ady;
        // level 0 holds cells in node form, so one word layout serves every
        // level; for a single cell the emptiness test below is exact (the
        // segment's z range [zlo, zhi] misses (-inf, h0] and [h1, h2] exactly
        // when zlo > top, or zlo > h0 and zhi < h1)
        const uint32_t word = cast_word<PAIR>(lv, level, nx, ny);
        if (STATS) {
            if (level > 0) cnt.nodes++;
            else cnt.cells++;
        }
        const int32_t maxh0 = word & 0xFF, minh1 = (word >> 8) & 0xFF,
                      maxtop = (word >> 16) & 0xFF;
        const bool down = r.dz < 0;
        const int32_t lo_num = down ? tout_num : tin_num, lo_den = down ? tout_den : tin_den;
        const int32_t hi_num = down ? tin_num : tout_num, hi_den = down ? tin_den : tout_den;
        const bool empty = zd(r.oz - (maxtop << kShift), r.dz, lo_num, lo_den) > 0 ||
                           (zd(r.oz - (maxh0 << kShift), r.dz, lo_num, lo_den) > 0 &&
                            zd(r.oz - (minh1 << kShift), r.dz, hi_num, hi_den) < 0);
        // advance past the node (or cell) through its exit side; at an exact
        // corner both indices change and the X face is reported
        auto advance = [&]() {
            if (cmp <= 0) nx += gx;
            if (cmp >= 0) ny += gy;
            entry = cmp <= 0 ? face_x : face_y;
            tin_num = tout_num;
            tin_den = tout_den;
            // ascend when the crossed boundary is a parent boundary: the new index
            // on the crossed axis is then even (odd for a negative direction)
            // (as arithmetic, not a branch: one control path for every lane)
            const int32_t crossed = cmp <= 0 ? (nx ^ qx) : (ny ^ qy);
            const int32_t up = (level < mip_start ? 1 : 0) & ~crossed & 1;
            level += up;
            nx >>= up;
            ny >>= up;
        };
        if (EMPTY_FIRST && empty) {
            advance();
            continue;
        }
        if (EMPTY_FIRST || !empty) {
            if (level > 0) {
                // descend into the child that holds the ray just after t_in:
                // the upper child on an axis when the ray has passed that
                // axis' midline by t_in (for a negative direction, when not)
                --level;
                const int32_t xm = (2 * nx + 1) * (1 << level), ym = (2 * ny + 1) * (1 << level);
                const int32_t midx = gx * (xm * (1 << kShift)) + kx;
                const int64_t lx = (int64_t)midx * tin_den;
                const int64_t rx = (int64_t)tin_num * adx;
                const int64_t ly = (int64_t)(gy * (ym * (1 << kShift)) + ky) * tin_den;
                const int64_t ry = (int64_t)tin_num * ady;
                nx = 2 * nx + ((lx <= rx) != (gx < 0) ? 1 : 0);
                ny = 2 * ny + ((ly <= ry) != (gy < 0) ? 1 : 0);
                // a corner: the ray enters the cell through its Y side and an
                // X cell boundary at the same instant; report the X face
                if (lx == rx && adx != 0 && entry == face_y) {
                    entry = face_x;
                    if (X_TIME) {
                        tin_num = midx;
                        tin_den = adx;
                    }
                }
                continue;
            }
            // a non-empty cell holds the hit (the cell test is exact: the
            // segment's z range meets (-inf, h0] or [h1, h2], and z is
            // continuous along it): find its layer, face and time.  The
            // advance is reached from empty nodes and cells only.
            if (!leaf_test(r.oz, r.dz, word, tin_num, tin_den, tout_num, tout_den, entry, h)) {
                h.face = kFaceError;  // (unreachable: the face would say so)
                h.layer = 255;
                return;
            }
            h.cx = nx;
            h.cy = ny;
            h.word = word;
            return;
        }
        advance();
    }
    h.face = kFaceError;
    h.layer = 255;
    cast_failed(status);
}

// The same as the warps of beams have it for a ray that no beam takes.
template <bool STATS, bool PAIR>
HF_HD void cast_general(const LevelDev *lvt, const Ray &r, int start_level, int mip_start,
                        int max_steps, Hit &h, Counters &cnt, uint32_t *status = nullptr) {
    cast_single<STATS, PAIR, true, true>((int32_t)lvt[0].stride, (int32_t)lvt[0].rows, lvt[0].base,
                                         lvt, r, start_level, mip_start, max_steps, status, h, cnt);
}

// One ray of a beam: a ray with a horizontal component, whose axis of the
// larger one (x on a tie) is u and whose other axis is v.  On an axis that the
// ray descends along, cell index n becomes ~n, so it always moves toward larger
// indices: a column (the cells of one u) is entered through its boundary u and
// left through u + 1, and on its way the ray crosses at most one boundary of v.
//
// The direction's part of it is the same for all rays toward one sun.
struct BeamDir {
    int32_t key;       // bit 2: u is x; bits 1, 0: u, v mirrored
    int32_t du, dv;    // |du|, |dv|
    float rho, sigma;  // rise of v and of the height per column, to a relative 2^-23
};
struct BeamRay {
    int32_t fu, fv;  // the start cell, mirrored
    int32_t ku, kv;  // minus the start's mirrored position, in 2^-16 units
    float z0;        // start height
    float pu, pv;    // the start relative to the beam's cell, v less a half (beam_place)
};

// (dx, dy not both 0)
HF_HD BeamDir beam_dir(int32_t dx, int32_t dy, int32_t dz) {
    BeamDir d;
    const int32_t ax = dx < 0 ? -dx : dx, ay = dy < 0 ? -dy : dy;
    const bool x_major = ax >= ay;
    const int32_t eu = x_major ? dx : dy, ev = x_major ? dy : dx;
    d.du = x_major ? ax : ay;
    d.dv = x_major ? ay : ax;
    d.key = (x_major ? 4 : 0) | (eu < 0 ? 2 : 0) | (ev < 0 ? 1 : 0);
    const float ru = cast_rcp((float)d.du);
    d.rho = (float)d.dv * ru;
    d.sigma = (float)dz * ru;
    return d;
}

HF_HD BeamRay beam_ray(const BeamDir &d, const Ray &r) {
    BeamRay q;
    const int32_t ou = d.key & 4 ? r.ox : r.oy, ov = d.key & 4 ? r.oy : r.ox;
    q.ku = d.key & 2 ? ou : -ou;
    q.kv = d.key & 1 ? ov : -ov;
    q.fu = (-q.ku) >> kShift;
    q.fv = (-q.kv) >> kShift;
    q.z0 = (float)r.oz * (1.0f / 65536.0f);
    return q;
}

HF_HD Ray beam_unray(const BeamDir &d, const BeamRay &q, int32_t oz, int32_t dz) {
    const int32_t ou = d.key & 2 ? q.ku : -q.ku, ov = d.key & 1 ? q.kv : -q.kv;
    const int32_t eu = d.key & 2 ? -d.du : d.du, ev = d.key & 1 ? -d.dv : d.dv;
    return d.key & 4 ? Ray{ou, ov, oz, eu, ev, dz} : Ray{ov, ou, oz, ev, eu, dz};
}

// A beam's rays, relative to the mirrored cell (u0, v0): at u = u0 + x every
// ray has v - v0 - 1/2 in [a0 + r0 x, a1 + r1 x] and a height between b0 + s0 x and
// b1 + s1 x, for x >= 0 (up to rounding, see beam_open).
struct Beam {
    int32_t u0, v0;
    float a0, a1, r0, r1, b0, b1, s0, s1;
};

// Takes a ray's start relative to the beam's cell: exact up to 256 cells, else
// rounded.  At u0 + x the ray is at v - v0 = 1/2 + pv + rho (x - pu) (so that the
// nearest integer to v - v0 - 1/2 is the row), and at the height z0 + sigma
// (x - pu); its terms of the beam are those at x = 0.
HF_HD void beam_place(BeamRay &q, const Beam &m) {
    q.pu = (float)(-q.ku - m.u0 * (1 << kShift)) * (1.0f / 65536.0f);
    q.pv = (float)(-q.kv - m.v0 * (1 << kShift) - (1 << (kShift - 1))) * (1.0f / 65536.0f);
}

// A bound of the error of a beam's heights up to x columns on: slopes have a
// relative error of 2^-23, and heights up to 4096 matter.  SAMPLES: of the heights of
// rounded samples, which lie up to kSampleAlong / 2 columns off their rays along u,
// and as far before the start (hf_march.h).
constexpr float kSampleAlong = 1.0f / 256.0f;
template <bool SAMPLES = false>
HF_HD float beam_slack(const Beam &m, float x) {
    float per = (fabsf(x) + 2.0f) * (1.0f / 1048576.0f);
    if (SAMPLES) per += kSampleAlong;
    return 0.02f + fmaxf(fabsf(m.s0), fabsf(m.s1)) * per;
}

// Whether the beam may meet a solid in mirrored columns [j 2^l, (j + 1) 2^l).
// The rows it covers there are read as nodes of level l.  high: their highest top.
template <bool PAIR, bool SAMPLES = false>
HF_HD bool beam_open(const LevelDev *lvt, const Beam &m, int l, int32_t j, int key,
                     uint32_t &high) {
    high = 0;
    const LevelDev lv = lvt[l];
    const bool x_major = key & 4;
    const uint32_t nu = x_major ? lv.stride : lv.rows, nv = x_major ? lv.rows : lv.stride;
    const uint32_t ju = (uint32_t)(key & 2 ? ~j : j);
    if (ju >= nu) return false;
    const float x0 = (float)(j * (1 << l) - m.u0), x1 = x0 + (float)(1 << l);
    const float zm = beam_slack<SAMPLES>(m, x1);
    const float zlo = m.b0 + fminf(m.s0 * x0, m.s0 * x1) - zm;
    const float zhi = m.b1 + fmaxf(m.s1 * x0, m.s1 * x1) + zm;
    // (rows, of samples too, are off by less than 2^-6 at the largest grid)
    const float vlo = m.a0 + fminf(m.r0 * x0, m.r1 * x0) + (0.5f - 0.015625f);
    const float vhi = m.a1 + m.r1 * x1 + (0.5f + 0.015625f);
    int32_t qa = (m.v0 + (int32_t)floorf(vlo)) >> l;
    int32_t qb = (m.v0 + (int32_t)floorf(vhi)) >> l;
    if (key & 1) {
        const int32_t c = ~qa;
        qa = ~qb;
        qb = c;
    }
    qa = qa < 0 ? 0 : qa;
    qb = qb < (int32_t)nv ? qb : (int32_t)nv - 1;
    uint32_t tops = 0, h1 = 0xFF00;  // highest top and floor, lowest slab
    for (int32_t jv = qa; jv <= qb; ++jv) {
        const uint32_t w = cast_word<PAIR>(lv, l, (int32_t)(x_major ? ju : jv),
                                           (int32_t)(x_major ? jv : ju));
        tops = max_halves(tops, w & 0xFF00FF);
        h1 = h1 < (w & 0xFF00) ? h1 : (w & 0xFF00);
    }
    high = tops >> 16;
    const float h0 = (float)(tops & 0xFF);
    return !(zlo > (float)high || (zlo > h0 && zhi < (float)(h1 >> 8)));
}

// A ray on its way through the columns of a run, up to x1 (columns x, rows and
// heights are relative to the beam's cell).
//
// Rows: v is off by less than ev = (x1 + |pu| + |pv| + 1) 1.5 2^-22: rho by
// 2^-23 of itself, x - pu, the start and the sum by 2^-24, and |rho| <= 1.  Where
// v is nearer than that to a boundary, the two are compared exactly; a ray through
// the corner itself is left to cast_general.
// Heights: off by less than e2 / 2 = (|sigma| (x1 + |pu| + 2) + |z0|) 2^-21.
struct BeamWalk {
    float ev, e2;
    float zbase;     // z0 - e2 / 2
    float zl;        // lower bound of the height where the column is entered
    int32_t row;     // the row it is entered in
};

enum { kBeamGoing = 0, kBeamOpen = 1, kBeamLeft = 2, kBeamCorner = 3 };

// The row (relative to m.v0) in which a ray enters column x of the beam.  False
// if it enters through a corner.
HF_HD bool beam_row(const BeamDir &d, const BeamRay &q, const Beam &m, const BeamWalk &w,
                    int32_t x, float dx, int32_t &row) {
    // rounding to the nearest integer by an addition: 3 2^22 has units of 1
    const float v = fmaf(d.rho, dx, q.pv), t = v + 12582912.0f, f = t - 12582912.0f;
    row = float_bits(t) - 0x4B400000;
    if (fabsf(v - f) < 0.5f - w.ev) return true;
    // which of the ray's crossings of the nearest row boundary and of column x
    // comes first
    row = (int32_t)floorf(v + 1.0f);
    const int64_t side = (int64_t)((m.v0 + row) * (1 << kShift) + q.kv) * d.du;
    const int64_t here = (int64_t)((m.u0 + x) * (1 << kShift) + q.ku) * d.dv;
    if (side > here) row -= 1;
    return side != here;
}

// Places a ray at column x0 of the run [x0, x1), or at its start if that lies
// beyond.  False if it enters through a corner.
HF_HD bool beam_enter(const BeamDir &d, const BeamRay &q, const Beam &m, int32_t x0, int32_t x1,
                      BeamWalk &w) {
    const float apu = fabsf(q.pu), far = (float)x1 + apu;
    w.ev = (far + fabsf(q.pv) + 1.0f) * (1.5f / 4194304.0f);
    const float e = (fabsf(d.sigma) * (far + 2.0f) + fabsf(q.z0)) * (1.0f / 2097152.0f);
    w.e2 = 2.0f * e;
    w.zbase = q.z0 - e;
    w.row = q.fv - m.v0;
    w.zl = fabsf(q.z0) < 256.0f ? q.z0 : w.zbase;  // (a start below 256 is exact)
    if (q.fu - m.u0 >= x0) return true;
    const float dx = (float)x0 - q.pu;
    w.zl = fmaf(d.sigma, dx, w.zbase);
    return beam_row(d, q, m, w, x0, dx, w.row);
}

// Word of cell index y W + x (pairs lie in one word: W is even).
template <bool PAIR>
HF_HD uint32_t beam_word(const uint32_t *cells, uint32_t cell) {
    return PAIR ? pair_node(cast_load(cells + (cell >> 1)), cell & 1) : cast_load(cells + cell);
}

// How mirrored rows and columns relative to the beam's cell lie in the grid:
// cell (x, row) has index at + x step_u + row step_v, and rows from `rows` on
// lie past the grid.
struct BeamGrid {
    const uint32_t *cells;
    uint32_t at;
    int32_t step_u, step_v, rows;
};
HF_HD BeamGrid beam_grid(const uint32_t *cells, const Beam &m, int key, uint32_t W, uint32_t H) {
    BeamGrid g;
    const bool x_major = key & 4;
    const uint32_t ru = (uint32_t)(key & 2 ? ~m.u0 : m.u0), rv = (uint32_t)(key & 1 ? ~m.v0 : m.v0);
    g.cells = cells;
    g.at = x_major ? rv * W + ru : ru * W + rv;
    g.step_u = (key & 2 ? -1 : 1) * (x_major ? 1 : (int32_t)W);
    g.step_v = (key & 1 ? -1 : 1) * (x_major ? (int32_t)W : 1);
    g.rows = (key & 1 ? 0 : (int32_t)(x_major ? H : W)) - m.v0;
    return g;
}

// A column of a walk: where it is left, and its one or two cells.
struct BeamColumn {
    int32_t row;      // the row it is left in
    float zl;         // lower bound of the height where it is left
    uint32_t wa, wb;  // words of the cells of the row it is entered in, and left in
};

// Column x of a walk, whose cells are tested together.  kBeamGoing: they are
// empty; kBeamOpen: they may not be; kBeamLeft: the ray has left the grid
// sideways; kBeamCorner: it leaves through a corner.
template <bool PAIR>
HF_HD int beam_step(const BeamGrid &g, const BeamDir &d, const BeamRay &q, const Beam &m,
                    const BeamWalk &w, int32_t x, BeamColumn &c) {
    if (w.row >= g.rows) return kBeamLeft;
    const float dx = (float)(x + 1) - q.pu;
    c.zl = fmaf(d.sigma, dx, w.zbase);
    const bool sure = beam_row(d, q, m, w, x + 1, dx, c.row);
    const uint32_t ca = g.at + (uint32_t)(x * g.step_u + w.row * g.step_v);
    const uint32_t cb = ca + (uint32_t)(c.row > w.row && c.row < g.rows ? g.step_v : 0);
    const uint32_t wa = beam_word<PAIR>(g.cells, ca), wb = beam_word<PAIR>(g.cells, cb);
    c.wa = wa;
    c.wb = wb;
    const uint32_t high = max_halves(wa & 0xFF00FF, wb & 0xFF00FF);  // top and floor
    const uint32_t ma = wa & 0xFF00, mb = wb & 0xFF00;
    const float top = (float)(high >> 16), h0 = (float)(high & 0xFF);
    const float h1 = (float)((ma < mb ? ma : mb) >> 8);
    const float zlo = fminf(w.zl, c.zl), zhi = fmaxf(w.zl, c.zl) + w.e2;
    if (!sure) return kBeamCorner;
    return (zlo > top) | ((zlo > h0) & (zhi < h1)) ? kBeamGoing : kBeamOpen;
}

// A hit as the walk finds it: mirrored cell (u, v), its word, and how it was hit.
enum { kBeamWallU = 0, kBeamWallV = 1, kBeamAbove = 2, kBeamBottom = 3, kBeamLayer1 = 4 };
struct BeamHit {
    int32_t u, v;
    uint32_t word;
    int32_t kind;  // the side it was entered through, with its layer; -1: no hit
};

// Decides a column that beam_step left open from the bounds of the heights where
// the ray enters it, changes row and leaves it.  The hit's kind, -1 if there is
// none, -2 if it is too close to tell.  second: it is in the row of the exit.
//
// The row changes where v = row + 1, at x - pu = (row + 1/2 - pv) / rho, off by
// less than 2 ev / rho.
HF_HD int beam_decide(const BeamGrid &g, const BeamDir &d, const BeamRay &q, const BeamWalk &w,
                      const BeamColumn &c, bool &second) {
    float il = w.zl, iu = w.zl + w.e2, ol = c.zl, ou = c.zl + w.e2;
    uint32_t word = c.wa;
    second = false;
    if (c.row > w.row) {
        const float inv = cast_rcp_fast(d.rho), es = fabsf(d.sigma) * (2.0f * w.ev) * inv;
        const float zs = fmaf(d.sigma, ((float)w.row + 0.5f - q.pv) * inv, w.zbase);
        const float sl = zs - es, su = zs + w.e2 + es;
        const float lo = fminf(il, sl), hi = fmaxf(iu, su);
        second = (lo > (float)(word >> 16 & 0xFF)) |
                 ((lo > (float)(word & 0xFF)) & (hi < (float)(word >> 8 & 0xFF)));
        if (second) {
            if (c.row >= g.rows) return -1;
            word = c.wb;
            il = sl;
            iu = su;
        } else {
            ol = sl;
            ou = su;
        }
    }
    const float h0 = (float)(word & 0xFF), h1 = (float)(word >> 8 & 0xFF),
                h2 = (float)(word >> 16 & 0xFF);
    const bool slab = h2 > h0;
    const bool gap = slab & (il > h0) & (iu < h1);
    if (iu <= h0) return second;
    if (slab & (il >= h1) & (iu <= h2)) return second + kBeamLayer1;
    if ((il > h2) & (ou <= h2)) return slab ? kBeamAbove + kBeamLayer1 : kBeamAbove;
    if (gap & (ou <= h0)) return kBeamAbove;
    if (gap & (ol >= h1)) return kBeamBottom + kBeamLayer1;
    const float lo = fminf(il, ol), hi = fmaxf(iu, ou);
    return (lo > h2) | ((lo > h0) & (hi < h1)) ? -1 : -2;
}

// The same on exact rationals: the hit's kind, or -1.  One column in two hundred
// comes here (beam_decide needs half of its instructions).
HF_HD int beam_exact(const BeamGrid &g, int32_t oz, int32_t dz, const BeamDir &d,
                     const BeamRay &q, const Beam &m, const BeamWalk &w, int32_t x,
                     const BeamColumn &c, bool &second) {
    const bool start = m.u0 + x == q.fu;
    const int32_t end = (m.u0 + x + 1) * (1 << kShift) + q.ku;        // over du: the column's exit
    const int32_t side = (m.v0 + w.row + 1) * (1 << kShift) + q.kv;   // over dv: the row's
    int32_t num = start ? 0 : end - (1 << kShift), den = start ? 1 : d.du;
    Hit h;
    for (second = false;; second = true) {
        const bool last = second || c.row == w.row;
        if (leaf_test(oz, dz, second ? c.wb : c.wa, num, den, last ? end : side,
                      last ? d.du : d.dv, kFaceInside, h))
            return (h.face == kFacePZ ? kBeamAbove : h.face == kFaceNZ ? kBeamBottom : second) +
                   (h.layer ? kBeamLayer1 : 0);
        if (last || c.row >= g.rows) return -1;
        num = side;
        den = d.dv;
    }
}

// Decides a column that beam_step left open: whether there is a hit, and h.
HF_HD bool beam_settle(const BeamGrid &g, int32_t oz, int32_t dz, const BeamDir &d,
                       const BeamRay &q, const Beam &m, const BeamWalk &w, int32_t x,
                       const BeamColumn &c, BeamHit &h) {
    bool second;
    int kind = beam_decide(g, d, q, w, c, second);
    if (kind < -1) kind = beam_exact(g, oz, dz, d, q, m, w, x, c, second);
    if (kind < 0) return false;
    h.u = m.u0 + x;
    h.v = m.v0 + w.row + second;
    h.word = second ? c.wb : c.wa;
    h.kind = kind;
    return true;
}

// The hit of a ray that has one.
HF_HD Hit beam_hit(const BeamHit &b, int32_t oz, int32_t dz, const BeamDir &d, const BeamRay &q) {
    Hit h;
    const bool x_major = d.key & 4;
    const int what = b.kind & 3;
    const bool top = what == kBeamAbove, level = what >= kBeamAbove;
    const bool on_v = what == kBeamWallV, start = what == kBeamWallU && b.u == q.fu;
    const int32_t ru = d.key & 2 ? ~b.u : b.u, rv = d.key & 1 ? ~b.v : b.v;
    h.cx = x_major ? ru : rv;
    h.cy = x_major ? rv : ru;
    h.word = b.word;
    h.layer = b.kind >> 2;
    // a face of x or y: the one that a mirrored ray enters through is the positive one
    const bool pos = d.key & (on_v ? 1 : 2);
    h.face = level ? (top ? kFacePZ : kFaceNZ)
             : start ? kFaceInside
                     : (x_major != on_v ? kFaceNX : kFaceNY) + (pos ? 1 : 0);
    const int32_t n = (top ? (h.layer ? b.word >> 16 : b.word) : b.word >> 8) & 0xFF;
    const int32_t fall = oz - (n << kShift);
    const int32_t at = (on_v ? b.v : b.u) * (1 << kShift) + (on_v ? q.kv : q.ku);
    h.tnum = level ? (top ? fall : -fall) : start ? 0 : at;
    h.tden = level ? (top ? -dz : dz) : start ? 1 : on_v ? d.dv : d.du;
    return h;
}

// The order in which a beam's columns are tested: rounds of 32 stretches of
// 2^level columns.  A round that finds nothing is followed by one of longer
// stretches, a long stretch that is open by a round of short ones from it on.
// kBeamLevel: 2-cell stretches; kBeamTop: what an empty beam climbs to.
// Open stretches that follow each other are walked as one.
// Rays that start more than kBeamSpread cells apart (along v, where they pass
// one column) are beams of their own.
constexpr int kBeamLevel = 1, kBeamTop = 5;
constexpr float kBeamSpread = 12.0f;

// How many stretches make the run at the lowest bit of open (not 0), bit i.
HF_HD int beam_run(uint32_t open, int i) {
    const uint32_t rest = ~(open >> i);
#ifdef __CUDA_ARCH__
    return rest ? __ffs((int)rest) - 1 : 32;
#else
    return rest ? __builtin_ctz(rest) : 32;
#endif
}

// The open stretches, with single closed ones between two of them: a march's run
// over such a gap costs less than two runs beside it (1.5 % over 384 renders;
// gaps of three stretches: no better than none, of seven or all: worse).
HF_HD uint32_t beam_joined(uint32_t open) { return open | (open << 1 & open >> 1); }

// The shortest stretches worth testing from u on: at least an eighth as long
// as the beam is wide there, so that one covers few nodes.
HF_HD int beam_least(const Beam &m, int32_t u, int base, int top) {
    const float wide = (m.a1 - m.a0) + (m.r1 - m.r0) * (float)(u - m.u0 + 64);
    int l = base;
    while (l < top && wide > (float)(8 << l)) ++l;
    return l;
}

// The first column to test, from u on: a beam that starts above every top
// is empty until its lowest ray comes down to them; one that rises above them
// is done (the limit is returned).  limit: the mirrored column past the grid.
template <bool SAMPLES = false>
HF_HD int32_t beam_skip(const Beam &m, int32_t u, int32_t limit, float top) {
    const float x0 = (float)(u - m.u0);
    if (!(m.b0 + m.s0 * x0 - beam_slack<SAMPLES>(m, x0) > top)) return u;
    if (m.s0 >= 0.0f) return limit;
    // where the lowest line is 0.04 above the top: it falls by at most 4096 up
    // to there, so it is off by less (and two columns are kept for a steep one)
    const float x = (top + 0.04f - m.b0) / m.s0;
    const float at = floorf(fminf(x, 40000.0f)) - 2.0f;
    const int32_t c = m.u0 + (int32_t)at;
    return c > u ? (c < limit ? c : limit) : u;
}

}  // namespace hf
