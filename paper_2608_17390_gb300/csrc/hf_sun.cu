// hf_sun.cu -- per-cell shadow bounds for one sun direction.
//
// Every shadow ray of a render runs along the same direction L (toward the
// sun), so what it can meet depends only on where it starts.  For each cell c
// two heights bound that in advance, for any origin in c (the cell the ray
// occupies just after t = 0, as the traversal picks it):
//
//   F(c): an origin at height z <= F is occluded.  Let u be the distance the
//         ray has travelled along the major axis of L (the axis with the
//         larger |L| component).  The ray enters the k-th column along that
//         axis after travelling at most k cells, so its height there is at
//         most z + k*Lz/|Lmaj|, and the row it enters lies in a band R_k of at
//         most three rows fixed by c and k.  If that height is at or below the
//         lowest floor of R_k, the cell it enters is solid at its entry time
//         (the floor has no lower bound, Section 3.1): a hit.  F is the best
//         such height over k (k = 0: the start cell's own floor), as long as
//         the band stays inside the grid (a ray that could leave the grid
//         sideways first proves nothing).
//
//   G(c): an origin at height z >= G is lit.  The ray rises, and it is in the
//         k-th column (k >= 1) only after travelling more than k - 1 cells,
//         so its height there exceeds z + (k-1)*Lz/|Lmaj|; every cell it can
//         occupy in that column lies in a band R'_k of at most four rows.  If
//         that bound is at or above every top (the highest solid point of a
//         cell) in R'_k, for every k, nothing is ever solid along the ray.
//
// Both bounds are exact rationals (scaled by |Lmaj|), rounded toward the safe
// side when stored: F down and G up, in units of 2^-8 world units, packed as
// F | G << 16 in one 32-bit word per cell.  A shadow ray whose origin lies at
// or below F is occluded and one at or above G is lit, with no traversal; any
// other is traced as before, so the shadow bit is the same as the flat cast's.
// The shadow map of the paper's shared shading path (Section 3) plays the same
// role -- sun visibility precomputed once per frame -- but approximately;
// these bounds only ever decide cases they prove.
//
// Only suns that rise (Lz > 0), are not vertical and clear the 255-unit
// height range within kSunMaxReach columns have bounds.  An edit of a
// rectangle changes the bounds of cells upstream of it (against L), within the
// distance over which a ray rises by 255 units: sun_bounds_region gives the
// rectangle that holds them, and sun_bounds_repair recomputes, inside it, the
// cells whose bands reach the edited rectangle (a parallelogram along L).
// The band rows and the rise depend on the column of travel only, not on the
// cell: a full build first tabulates them (k_sun_rows) after the bounds words,
// and the build and later repairs read the table instead of dividing.
#include <cuda_runtime.h>

#include <cstdint>

#include "hf.h"
#include "hf_internal.h"

namespace hf {
namespace {

// A table after the bounds words, one entry per column of major travel, set by
// one pass per sun.  Entry i = k + 2, k = -2 .. kRowTable - 3:
//   x:  q(k + 1), where q(j) = floor(lmin j / lmaj), the minor-axis rows a ray
//       has crossed after j columns;
//   y:  ceil of 256 k lz / lmaj, and z: floor of 256 (k - 1) lz / lmaj, its
//       rise in the bounds' units (2^-8 world units), saturated at kRiseSat
//       (every quantity it is compared with is below 2^17, so saturation
//       changes no outcome).
constexpr int32_t kRiseSat = 1 << 21;

constexpr int kSunThreads = 128;
// Cells of a thread along the minor axis.  Their bands overlap, so V cells read
// V + 3 words a column instead of 4 V.  x major: the lanes of a warp lie along
// the major axis and every load is one row of words (4; 2 cost 12 % more, 8 the
// same); y major: along the minor axis, where V also spreads a warp's loads (2).
constexpr int kSunCellsX = 4, kSunCellsY = 2;
// Up to this many groups of 32 threads, 8 warps share a group's columns: a
// repair after a crater, or a small world, leaves too few groups to hide the
// latency of a thread's up to 1056 columns one after the other (a repair toward
// (400000, 100000, 100000) 0.143 -> 0.084 ms with its edit; a 2048^2 build, 32768
// groups, took two thirds longer if split, as each warp then stops later).
constexpr int kSunSplit = 8;
// Columns of a round are read in parts of 16, and a part over a region whose
// nodes of 8 x 8 cells show nothing high enough is left out: two 2048^2 builds and
// 1080p views 1331 -> 1254 us (parts of 8: 1282; of 16 over 16 x 16 nodes: 1.5 % more).
constexpr int kSunPart = 16, kSunPartLevel = 3;
constexpr uint32_t kSunSplitBelow = 16384;

// The table's entries.  No column past K + 1, K = kSunMaxReach, can raise a bound
// (sun_bounds_eligible), so none is looked into: the last round that is ends at
// column K + 32 and asks for the rows after K + 33, entry K + 34; a split warp's next
// part starts up to kSunPart * kSunSplit columns further on, and is looked up, entry
// k + 2, before it is left out.
constexpr int kRowTable = (int)kSunMaxReach + kSunPart * kSunSplit + 64;
static_assert(kRowTable > (int)kSunMaxReach + 1 + kSunPart * kSunSplit + 2 &&
                  kRowTable > (int)kSunMaxReach + 1 + 32 + 1,
              "every column that a bound may ask for has its entry");

__global__ void k_sun_rows(int4 *tab, int64_t lmin, int64_t lmaj, int64_t lz) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= kRowTable) return;
    // once per sun: exact divisions are affordable here
    auto floor_div = [](int64_t n, int64_t d) {
        int64_t f = n / d;
        if (n % d != 0 && n < 0) f -= 1;
        return f;
    };
    const int64_t k = i - 2;
    const int64_t up = -floor_div(-256 * k * lz, lmaj), down = floor_div(256 * (k - 1) * lz, lmaj);
    tab[i] = make_int4((int32_t)floor_div(lmin * (k + 1), lmaj), (int32_t)min(up, (int64_t)kRiseSat),
                       (int32_t)min(down, (int64_t)kRiseSat), 0);
}

// Words of the bounds, rounded up to whole table entries.
__host__ __device__ __forceinline__ size_t sun_words(int32_t W, int32_t H) {
    return ((size_t)W * (size_t)H + 3) & ~(size_t)3;
}

struct SunAxes {
    int32_t lmaj;   // |L| along the major axis (> 0)
    int32_t lmin;   // signed L along the minor axis
    int32_t lz;     // > 0
    int32_t smaj;   // +1 / -1: direction along the major axis
    bool x_major;   // the major axis is x
};

// q(j) = floor(lmin j / lmaj), j >= -1
__device__ __forceinline__ int32_t rows_after(const int4 *tab, int32_t j) {
    return __ldg(&tab[j + 1].x);
}

// A level-0 cell as the bounds use it: 255 - floor in the low half, top in the
// high half, so that one 16-bit pairwise maximum over a band's cells gives its
// lowest floor and its highest top.
//
// `at` is 4 (y W + x), the byte at which the cell's word starts: a 32-bit offset
// from one pointer (a world has at most 2^28 cells) that the load adds itself.
// With a 64-bit address per load a 2048^2 build with the default sun took 0.47
// ms instead of 0.41.
template <bool PAIR>
__device__ __forceinline__ uint32_t sun_cell(const WorldDev &w, uint32_t at) {
    const char *base = reinterpret_cast<const char *>(w.base);
    const uint32_t word = __ldg(reinterpret_cast<const uint32_t *>(base + (PAIR ? at >> 1 & ~3u : at)));
    return ((PAIR ? pair_node(word, at >> 2 & 1) : word) ^ 0xFFu) & 0x00FF00FFu;
}

// V cells of one thread, next to each other along the minor axis in the
// direction of the sun's minor component: cell i lies at minor coordinate
// cv + sv i.
//
// Column k of a cell reads the band of rows j = 0 .. 1 + B from row(k) =
// cv + sv i + (sv > 0 ? q(k - 1) : 1 + q(k - 1)) on, in direction sv: the rows
// 0 .. 1 + A for F, all of them for G, A = |q(k) - q(k - 1)| <= 1 and
// B = |q(k + 1) - q(k - 1)| <= A + 1.  So the V cells share V + 1 + B rows.
// F and G are kept times 256, so that a term is a cell's byte, shifted, plus the
// column's rise: one add with maximum (and for F one multiplication that takes
// the low half of the band's maximum; for G the low half only adds less than a
// unit, which the final shift drops).
template <int V>
struct SunCells {
    int32_t F[V], G[V];
};

// One column: col, row: its major coordinate and the first cell's row(k).
// EDGE: some of it may lie outside the grid (a cell there is neutral); f_on:
// cells whose F still counts.
template <bool XM, bool PAIR, int V, int A, int B, bool EDGE>
__device__ __forceinline__ void sun_column(const WorldDev &w, int32_t col, int32_t row, int32_t sv,
                                           int32_t up, int32_t down, uint32_t f_on,
                                           SunCells<V> &c) {
    const int32_t NU = XM ? w.W : w.H, NV = XM ? w.H : w.W;
    const bool in_col = !EDGE || (uint32_t)col < (uint32_t)NU;
    uint32_t p[V + 1 + B];
    const uint32_t at = 4u * (uint32_t)(XM ? row * w.W + col : col * w.W + row);
    const uint32_t per_row = 4u * (uint32_t)(XM ? sv * w.W : sv);
#pragma unroll
    for (int j = 0; j < V + 1 + B; ++j) {
        p[j] = 0;
        if (!EDGE || (in_col && (uint32_t)(row + sv * j) < (uint32_t)NV))
            p[j] = sun_cell<PAIR>(w, at + (uint32_t)j * per_row);
    }
    const int32_t cf = ((255 << 8) - up) * 256, cg = -down * 256;
#pragma unroll
    for (int i = 0; i < V; ++i) {
        const uint32_t f = A ? __vimax3_u16x2(p[i], p[i + 1], p[i + 1 + A]) : __vmaxu2(p[i], p[i + 1]);
        const uint32_t g = B > A ? __vmaxu2(f, p[i + 1 + B]) : f;
        // the whole F band in the grid
        const bool f_ok = !EDGE || (in_col && (f_on >> i & 1) &&
                                    (uint32_t)(row + sv * i) < (uint32_t)NV &&
                                    (uint32_t)(row + sv * (i + 1 + A)) < (uint32_t)NV);
        if (f_ok) c.F[i] = __viaddmax_s32((int32_t)(f * 0xFFFF0000u), cf, c.F[i]);
        c.G[i] = __viaddmax_s32((int32_t)g, cg, c.G[i]);  // (never raised by neutral cells)
    }
}

template <bool XM, bool PAIR, int V, bool EDGE>
__device__ __forceinline__ void sun_part(const WorldDev &w, const SunAxes &a, const int4 *tab,
                                          int32_t k0, int32_t cu, int32_t cv, int32_t sv,
                                          uint32_t f_on, SunCells<V> &c) {
    int32_t qm = rows_after(tab, k0 - 1), qk = rows_after(tab, k0);
#pragma unroll 1
    for (int32_t k = k0; k < k0 + kSunPart; ++k) {
        const int4 e = __ldg(&tab[k + 2]);
        const int32_t col = cu + a.smaj * k, row = cv + (sv > 0 ? qm : 1 + qm);
        if (qk != qm) {
            if (abs(e.x - qm) > 1)
                sun_column<XM, PAIR, V, 1, 2, EDGE>(w, col, row, sv, e.y, e.z, f_on, c);
            else
                sun_column<XM, PAIR, V, 1, 1, EDGE>(w, col, row, sv, e.y, e.z, f_on, c);
        } else {
            if (e.x != qm)
                sun_column<XM, PAIR, V, 0, 1, EDGE>(w, col, row, sv, e.y, e.z, f_on, c);
            else
                sun_column<XM, PAIR, V, 0, 0, EDGE>(w, col, row, sv, e.y, e.z, f_on, c);
        }
        qm = qk;
        qk = e.x;
    }
}

// Whether a floor or top in region [u0, u1] x [v0, v1] (it meets the grid) can
// raise a bound: the highest there, from the nodes of a level, against the
// lowest bounds and the rise in the region's first column.
template <bool XM>
__device__ __forceinline__ bool sun_may_rise(const WorldDev &w, int level, int32_t u0, int32_t u1,
                                             int32_t v0, int32_t v1, int32_t lo_f, int32_t lo_g,
                                             int32_t up, int32_t down) {
    // lanes side by side along the region's longer axis
    constexpr int kU = XM ? 8 : 2, kV = 32 / kU;
    const int32_t NU = XM ? w.W : w.H, NV = XM ? w.H : w.W;
    const int lane = threadIdx.x & 31;
    const int32_t a1 = min(u1, NU - 1) >> level, b1 = min(v1, NV - 1) >> level;
    const uint32_t *nodes = w.base + w.off[level];
    const uint32_t stride = w.stride[level];
    uint32_t top = 0, h0 = 0;
    for (int32_t u = (max(u0, 0) >> level) + lane % kU; u <= a1; u += kU)
        for (int32_t v = (max(v0, 0) >> level) + lane / kU; v <= b1; v += kV) {
            const uint32_t n = __ldg(nodes + (uint32_t)(XM ? v : u) * stride + (uint32_t)(XM ? u : v));
            top = max(top, n & 0xFF0000u);
            h0 = max(h0, n & 0xFFu);
        }
    const int32_t mt = (int32_t)(__reduce_max_sync(0xFFFFFFFFu, top) >> 8);
    const int32_t mh = (int32_t)(__reduce_max_sync(0xFFFFFFFFu, h0) << 8);
    return mh - (lo_f + 1) >= up || mt - lo_g > down;
}

// Bounds of the V cells of each thread of a warp, rounded to the stored units
// (F down, G up, 2^-8 world units).  In these units a term is a height h times
// 256, less the rise: exactly, the F term of column k rounded down is 256 h -
// ceil(256 k lz / lmaj), and the G term rounded up is 256 h - floor(256 (k - 1)
// lz / lmaj).
//
// Columns go in rounds of 32, each in parts of kSunPart.  F stops with the first
// round that holds a column it cannot use (the grid's end, or a band that leaves
// the grid: once one does, all later ones do too, but for column 1 of a cell on
// the grid's last row).  The parts end once none can raise any of the warp's
// bounds (maxh0, maxtop: the world's highest floor and top), and a round or part
// over a region whose highest floor and top (of its level-5 nodes, of its nodes
// of kSunPartLevel) cannot raise any is skipped; neither changes a bound.  SPLIT:
// this warp takes every kSunSplit-th part from `first` on (and not whole rounds:
// with 10 rounds for 8 warps, two of them would have twice the work).
// cu, cv: the first cell; on: which cells are real.
template <bool XM, bool PAIR, int V, bool SPLIT>
__device__ __forceinline__ void sun_bounds_of(const WorldDev &w, const SunAxes &a, const int4 *tab,
                                              int32_t cu, int32_t cv, int32_t sv, uint32_t on,
                                              int32_t first, SunCells<V> &c) {
    constexpr unsigned full = 0xFFFFFFFFu;
    const int32_t NU = XM ? w.W : w.H, NV = XM ? w.H : w.W;
    auto cell = [&](int32_t u, int32_t v) {
        return sun_cell<PAIR>(w, 4u * (uint32_t)(XM ? v * w.W + u : u * w.W + v));
    };
    // k = 0: for F the start cell's floor; for G the rows the ray can cross in
    // its start column (it moves at most one row there), strictly above: top +
    // 2^-16, rounded up
#pragma unroll
    for (int i = 0; i < V; ++i) {
        c.F[i] = c.G[i] = 0;
        if (!(on >> i & 1)) continue;
        const int32_t v = cv + sv * i;
        const uint32_t p = cell(cu, v);
        uint32_t top = p >> 16;
        if (v + 1 < NV) top = max(top, cell(cu, v + 1) >> 16);
        if (a.lmin < 0 && v > 0) top = max(top, cell(cu, v - 1) >> 16);
        c.F[i] = (int32_t)(255 - (p & 0xFF)) << 16;
        c.G[i] = ((int32_t)(top << 8) + 1) << 8;
    }
    const uint32_t root = __ldg(w.base + w.off[w.L]);
    const int32_t maxh0 = w.L ? (int32_t)(root & 0xFF) << 8 : 255 << 8;
    const int32_t maxtop = w.L ? (int32_t)((root >> 16) & 0xFF) << 8 : 255 << 8;
    // cells whose F band leaves the grid in column k
    auto f_out = [&](int32_t k) {
        const int32_t qa = rows_after(tab, k - 1), qb = rows_after(tab, k);
        const int32_t col = cu + a.smaj * k;
        uint32_t out = 0;
#pragma unroll
        for (int i = 0; i < V; ++i) {
            const int32_t v = cv + sv * i;
            if (col < 0 || col >= NU || v + min(qa, qb) < 0 || v + 1 + max(qa, qb) >= NV)
                out |= 1u << i;
        }
        return out;
    };
    const uint32_t out1 = f_out(1);
    int32_t lo_f, lo_g;  // the lowest bounds that may still rise
    auto lowest = [&](uint32_t f_on) {
        lo_f = lo_g = 1 << 28;
#pragma unroll
        for (int i = 0; i < V; ++i) {
            if (f_on >> i & 1) lo_f = min(lo_f, c.F[i]);
            if (on >> i & 1) lo_g = min(lo_g, c.G[i]);
        }
        lo_f = __reduce_min_sync(full, lo_f) >> 8;
        lo_g = __reduce_min_sync(full, lo_g) >> 8;
    };
    // what the warp reads in columns [k, k + n): first and last of each axis
    int32_t u0, u1, v0, v1;
    auto region = [&](int32_t k, int32_t n) {
        const int32_t ca = cu + a.smaj * k, cb = cu + a.smaj * (k + n - 1);
        // the first and the last row in direction sv
        const int32_t qm = rows_after(tab, k - 1), qe = rows_after(tab, k + n);
        const int32_t ra = cv + (sv > 0 ? qm : 1 + qm);
        const int32_t rb = cv + sv * (V - 1) + (sv > 0 ? 1 + qe : qe);
        u0 = __reduce_min_sync(full, min(ca, cb));
        u1 = __reduce_max_sync(full, max(ca, cb));
        v0 = __reduce_min_sync(full, min(ra, rb));
        v1 = __reduce_max_sync(full, max(ra, rb));
        return u1 >= 0 && u0 < NU && v1 >= 0 && v0 < NV;  // it meets the grid
    };
    // f_on: cells whose F band was in the grid up to the round of column k
    uint32_t f_on = on;
#pragma unroll 1
    for (int32_t k = 1 + (SPLIT ? kSunPart * first : 0);;
         k += SPLIT ? kSunPart * kSunSplit : kSunPart) {
        const bool round = (k - 1) % 32 == 0;
        if (SPLIT || round) {
            const int32_t k0 = (k - 1) / 32 * 32 + 1;
            f_on = k0 == 1 ? on : on & ~(out1 | f_out(k0 - 1));
        }
        lowest(f_on);
        const int4 rise = __ldg(&tab[k + 2]);
        if (maxh0 - (lo_f + 1) < rise.y && maxtop - lo_g <= rise.z) break;
        if (!SPLIT && round && w.L >= 5) {
            if (!region(k, 32)) break;  // and so do all later rounds
            if (!sun_may_rise<XM>(w, 5, u0, u1, v0, v1, lo_f, lo_g, rise.y, rise.z)) {
                k += 32 - kSunPart;
                continue;
            }
        }
        if (!region(k, kSunPart)) break;
        if (w.L >= kSunPartLevel &&
            !sun_may_rise<XM>(w, kSunPartLevel, u0, u1, v0, v1, lo_f, lo_g, rise.y, rise.z))
            continue;
        if (u0 >= 0 && u1 < NU && v0 >= 0 && v1 < NV && __all_sync(full, f_on == on))
            sun_part<XM, PAIR, V, false>(w, a, tab, k, cu, cv, sv, f_on, c);
        else
            sun_part<XM, PAIR, V, true>(w, a, tab, k, cu, cv, sv, f_on, c);
    }
}

// Whether the bounds of cell (cu, cv) read any cell of the rectangle
// [eu0, eu1) x [ev0, ev1) (major / minor coordinates): some column of the
// rectangle within `reach` columns downstream, with the cell's widest band
// over those columns meeting the rectangle's rows.
__device__ bool depends_on(const SunAxes &a, const int4 *tab, int32_t cu, int32_t cv,
                           int32_t eu0, int32_t ev0, int32_t eu1, int32_t ev1, int32_t reach) {
    int32_t ka = a.smaj > 0 ? eu0 - cu : cu - (eu1 - 1);
    int32_t kb = a.smaj > 0 ? eu1 - 1 - cu : cu - eu0;
    ka = max(ka, 0);
    kb = min(kb, reach);
    if (ka > kb) return false;
    // floor is monotone, so the band's lowest and highest rows over the
    // columns ka..kb come from travel ka - 1 and kb + 1
    const int32_t qa = rows_after(tab, ka - 1), qb = rows_after(tab, kb + 1);
    return cv + 1 + max(qa, qb) >= ev0 && cv + min(qa, qb) < ev1;
}

// Bound by instruction issue (about 10 instructions per cell and column).  One
// warp per cell, its lanes taking 32 columns each round, cost about 1700 warp
// instructions a cell in loads of bands no other cell shared, reductions and
// per-lane table reads: 2048^2 world, default sun, 6.4 -> 0.40 ms.
// The cells of the rectangle [x0, x1) x [y0, y1), V per thread along the minor
// axis, a warp's threads next to each other along x (nwx warps a row).  SPLIT:
// the warps of a block share the rounds of the same cells.  With edit.z >
// edit.x, only the cells whose bounds depend on the edited rectangle [edit.x,
// edit.z) x [edit.y, edit.w) are recomputed (the others keep theirs).
template <bool XM, bool PAIR, int V, bool SPLIT>
__global__ void __launch_bounds__(SPLIT ? kSunSplit * 32 : kSunThreads)
    k_sun_bounds(const WorldDev w, uint32_t *fg, const SunAxes a, int32_t x0, int32_t y0, int32_t x1,
                 int32_t y1, uint32_t nwx, uint32_t n_groups, int4 edit, int32_t reach) {
    __shared__ int32_t s_part[SPLIT ? 2 * V * kSunSplit * 32 : 1];
    const uint32_t group = SPLIT ? blockIdx.x : (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (group >= n_groups) return;
    const int lane = threadIdx.x & 31, sub = SPLIT ? threadIdx.x >> 5 : 0;
    const int4 *tab = reinterpret_cast<const int4 *>(fg + sun_words(w.W, w.H));
    const int32_t sv = a.lmin < 0 ? -1 : 1;
    const int32_t wx = (int32_t)(group % nwx), wy = (int32_t)(group / nwx);
    // the thread's first cell along the minor axis, and its major coordinate
    const int32_t v0 = XM ? y0 + wy * V : x0 + (wx * 32 + lane) * V, v1 = XM ? y1 : x1;
    const int32_t u = XM ? x0 + wx * 32 + lane : y0 + wy;
    const int32_t cu = XM ? min(u, x1 - 1) : u;
    const int32_t cv = min(v0, v1 - 1) + (sv < 0 ? V - 1 : 0);
    uint32_t on = 0;
    if (v0 < v1 && (!XM || u < x1))
        for (int i = 0; i < V; ++i) {
            const int32_t v = cv + sv * i;
            if (v >= v1) continue;
            if (edit.z > edit.x &&
                !(XM ? depends_on(a, tab, cu, v, edit.x, edit.y, edit.z, edit.w, reach)
                     : depends_on(a, tab, cu, v, edit.y, edit.x, edit.w, edit.z, reach)))
                continue;
            on |= 1u << i;
        }
    if (!__any_sync(0xFFFFFFFFu, on != 0)) return;  // (all warps of a split group alike)
    SunCells<V> c;
    sun_bounds_of<XM, PAIR, V, SPLIT>(w, a, tab, cu, cv, sv, on, sub, c);
    if (SPLIT) {
#pragma unroll
        for (int i = 0; i < V; ++i) {
            s_part[(2 * i * kSunSplit + sub) * 32 + lane] = c.F[i];
            s_part[((2 * i + 1) * kSunSplit + sub) * 32 + lane] = c.G[i];
        }
        __syncthreads();
        if (sub) return;
#pragma unroll
        for (int i = 0; i < V; ++i)
            for (int t = 1; t < kSunSplit; ++t) {
                c.F[i] = max(c.F[i], s_part[(2 * i * kSunSplit + t) * 32 + lane]);
                c.G[i] = max(c.G[i], s_part[((2 * i + 1) * kSunSplit + t) * 32 + lane]);
            }
    }
#pragma unroll
    for (int i = 0; i < V; ++i) {
        if (!(on >> i & 1)) continue;
        const int32_t v = cv + sv * i;
        fg[(uint32_t)(XM ? v : cu) * (uint32_t)w.W + (uint32_t)(XM ? cu : v)] =
            (uint32_t)(c.F[i] >> 8) | ((uint32_t)(c.G[i] >> 8) << 16);
    }
}

template <bool XM, bool PAIR, int V>
int sun_launch(const WorldDev &w, uint32_t *fg, const SunAxes &a, const int32_t r[4], int4 edit,
               int32_t reach, cudaStream_t s) {
    const uint32_t nx = (uint32_t)(r[2] - r[0]), ny = (uint32_t)(r[3] - r[1]);
    const uint32_t per = XM ? 32 : 32 * V, nwx = (nx + per - 1) / per;
    const uint32_t n = nwx * (XM ? (ny + V - 1) / V : ny);
    if (n <= kSunSplitBelow)
        k_sun_bounds<XM, PAIR, V, true><<<n, kSunSplit * 32, 0, s>>>(w, fg, a, r[0], r[1], r[2], r[3],
                                                                     nwx, n, edit, reach);
    else
        k_sun_bounds<XM, PAIR, V, false>
            <<<(n * 32 + kSunThreads - 1) / kSunThreads, kSunThreads, 0, s>>>(
                w, fg, a, r[0], r[1], r[2], r[3], nwx, n, edit, reach);
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

int sun_launch(const WorldDev &w, uint32_t *fg, const SunAxes &a, const int32_t r[4], int4 edit,
               int32_t reach, cudaStream_t s) {
    if (a.x_major)
        return w.pair ? sun_launch<true, true, kSunCellsX>(w, fg, a, r, edit, reach, s)
                      : sun_launch<true, false, kSunCellsX>(w, fg, a, r, edit, reach, s);
    return w.pair ? sun_launch<false, true, kSunCellsY>(w, fg, a, r, edit, reach, s)
                  : sun_launch<false, false, kSunCellsY>(w, fg, a, r, edit, reach, s);
}

SunAxes axes_of(const int32_t sun[3]) {
    SunAxes a;
    const int32_t ax = sun[0] < 0 ? -sun[0] : sun[0], ay = sun[1] < 0 ? -sun[1] : sun[1];
    a.x_major = ax >= ay;
    a.lmaj = a.x_major ? ax : ay;
    a.lmin = a.x_major ? sun[1] : sun[0];
    a.smaj = (a.x_major ? sun[0] : sun[1]) < 0 ? -1 : 1;
    a.lz = sun[2];
    return a;
}

}  // namespace

bool sun_bounds_eligible(const int32_t sun[3]) {
    if (sun[2] <= 0 || (sun[0] == 0 && sun[1] == 0)) return false;
    const SunAxes a = axes_of(sun);
    // the columns a ray crosses before it has risen by 255 units: the work
    // per cell grows with it, so suns lower than this are traced instead
    return 255 * (int64_t)a.lmaj / a.lz + 2 <= kSunMaxReach;
}

void sun_bounds_region(const WorldDev &w, const int32_t sun[3], int32_t x0, int32_t y0,
                       int32_t x1, int32_t y1, int32_t *out) {
    const SunAxes a = axes_of(sun);
    // beyond K columns a ray has risen past every top: no term there matters
    const int64_t K = 255 * (int64_t)a.lmaj / a.lz + 2;
    const int64_t D = (int64_t)(a.lmin < 0 ? -a.lmin : a.lmin) * (K + 1) / a.lmaj + 2;
    int64_t u0 = a.x_major ? x0 : y0, u1 = a.x_major ? x1 : y1;
    int64_t v0 = a.x_major ? y0 : x0, v1 = a.x_major ? y1 : x1;
    if (a.smaj > 0) u0 -= K;  // upstream: cells whose rays run into the rectangle
    else u1 += K;
    v0 -= D;
    v1 += D;
    const int64_t NU = a.x_major ? w.W : w.H, NV = a.x_major ? w.H : w.W;
    u0 = u0 < 0 ? 0 : u0;
    v0 = v0 < 0 ? 0 : v0;
    u1 = u1 > NU ? NU : u1;
    v1 = v1 > NV ? NV : v1;
    out[0] = (int32_t)(a.x_major ? u0 : v0);
    out[1] = (int32_t)(a.x_major ? v0 : u0);
    out[2] = (int32_t)(a.x_major ? u1 : v1);
    out[3] = (int32_t)(a.x_major ? v1 : u1);
}

size_t sun_bounds_bytes(int32_t W, int32_t H) {
    return sun_words(W, H) * sizeof(uint32_t) + kRowTable * sizeof(int4);
}

int sun_bounds(const WorldDev &w, uint32_t *fg, const int32_t sun[3], int32_t x0, int32_t y0,
               int32_t x1, int32_t y1, void *stream) {
    if (!sun_bounds_eligible(sun)) return -1;
    const SunAxes a = axes_of(sun);
    // this sun's table, which the bounds and later repairs read
    k_sun_rows<<<(kRowTable + 127) / 128, 128, 0, (cudaStream_t)stream>>>(
        reinterpret_cast<int4 *>(fg + sun_words(w.W, w.H)), a.lmin, a.lmaj, a.lz);
    if (cudaGetLastError() != cudaSuccess) return -1;
    if (x1 <= x0 || y1 <= y0) return 0;
    const int32_t r[4] = {x0, y0, x1, y1};
    return sun_launch(w, fg, a, r, make_int4(0, 0, 0, 0), 0, (cudaStream_t)stream);
}

int sun_bounds_repair(const WorldDev &w, uint32_t *fg, const int32_t sun[3], int32_t x0,
                      int32_t y0, int32_t x1, int32_t y1, void *stream) {
    if (!sun_bounds_eligible(sun)) return -1;
    if (x1 <= x0 || y1 <= y0) return 0;
    int32_t r[4];
    sun_bounds_region(w, sun, x0, y0, x1, y1, r);
    if (r[2] <= r[0] || r[3] <= r[1]) return 0;
    const SunAxes a = axes_of(sun);
    const int32_t reach = (int32_t)(255 * (int64_t)a.lmaj / a.lz + 2);
    return sun_launch(w, fg, a, r, make_int4(x0, y0, x1, y1), reach, (cudaStream_t)stream);
}

}  // namespace hf
