// hf_voxel.cu -- the paper's voxel-accelerated ray march, RayVoxel (its
// Section 3), as a comparison renderer: a conservative occupancy pyramid and a
// hierarchical DDA with fixed sampling at the leaves.
//
// Occupancy.  Level-0 voxel (i, j, k) covers cells [i vx, (i+1) vx) x
// [j vy, (j+1) vy) and heights [k vz, (k+1) vz] (closed); it is occupied when
// some cell there is solid at some such height (z0 <= h0, or a slab with
// h1 <= z1 and z0 <= h2).  Level l+1 voxel = OR of its eight level-l children.
// Each level is stored as Morton-coded 8 x 8 x 8 tiles of bits: tile
// (tx, ty, tz) at (tz TY + ty) TX + tx, 16 words of 32 bits each, voxel bit
// morton3(x & 7, y & 7, z & 7) (bits of x, y, z interleaved from the lowest).
//
// Traversal (one thread per pixel; float32, round to nearest, no fused
// multiply-add, in a fixed order, so results are reproducible bit for bit):
// clip the ray to the voxel grid's box and the far distance; start at the top
// level; an empty voxel advances to its exit plane (climbing a level when the
// crossed plane is a parent boundary); an occupied one is opened (the child
// the ray is in just after t: the first child along the direction on the axis
// last crossed, else the one holding p(t)); an occupied leaf is sampled at
// `inner` midpoints of the ray's stretch inside it, and the first SOLID sample
// is the hit.  Thin features can slip between samples (the paper's trade-off).
#include <cuda_runtime.h>

#include "hf_internal.h"

namespace hf {
namespace {

constexpr int kVoxThreads = 128;
constexpr int kVoxMinBlocks = 8;  // trace blocks per SM (56 registers; 10 with 48: 6 % slower)
constexpr int kVoxTailThreads = 1024;
constexpr int32_t kVoxTailWords = 16384;  // levels of up to this many words share one block

// Bits 0, 1, 2 of v at 0, 3, 6: byte v & 7 of a table of eight.
__device__ __forceinline__ uint32_t spread3(uint32_t v) {
    return __byte_perm(0x09080100u, 0x49484140u, v & 7);
}
__device__ __forceinline__ uint32_t morton3(uint32_t x, uint32_t y, uint32_t z) {
    return spread3(x) | (spread3(y) << 1) | (spread3(z) << 2);
}

// One level of the pyramid as the traversal reads it: a per-block shared
// table, so lanes at different levels read it in one shared-memory access
// (kernel parameters indexed by a per-lane level would serialise).
struct __align__(16) VoxLevel {
    uint32_t off;
    int32_t tx, ty, pad0;
    int32_t n[3], pad1;
};

__device__ __forceinline__ bool vox_occupied(const VoxelDev &v, const VoxLevel &lv, uint32_t x,
                                             uint32_t y, uint32_t z) {
    const uint32_t tile = ((z >> 3) * (uint32_t)lv.ty + (y >> 3)) * (uint32_t)lv.tx + (x >> 3);
    const uint32_t m = morton3(x, y, z);
    return (__ldg(v.words + lv.off + tile * 16 + (m >> 5)) >> (m & 31)) & 1u;
}

// leaf sample fractions (s + 0.5) / inner held in shared memory up to this count
constexpr int kVoxFracTable = 64;

// log2 of a power-of-two voxel extent, else -1
__host__ __device__ __forceinline__ int32_t pow2_log2(int32_t v) {
    if (v <= 0 || (v & (v - 1))) return -1;
    int32_t e = 0;
    while ((1 << e) < v) ++e;
    return e;
}

// The correctly rounded quotient pk / (vs 2^l).  For a power-of-two extent
// (vs = 2^e) it is the correctly rounded product pk 2^-(e+l): both round the
// same real number, and 2^-(e+l) (at least 2^-21) is an exact float.
__device__ __forceinline__ float vox_quot(float pk, int32_t vs, int32_t vs_log2, int l) {
    if (vs_log2 >= 0) return __fmul_rn(pk, __int_as_float((127 - vs_log2 - l) << 23));
    return __fdiv_rn(pk, (float)(vs << l));
}

// h / vz for h < 512, vz <= 256, by a multiplication with recip = 2^20 / vz + 1
// (the product's excess, h (recip vz - 2^20) <= 2^17, stays below 2^20).
__device__ __forceinline__ int32_t vox_div(int32_t h, uint32_t recip) {
    return (int32_t)(((uint32_t)h * recip) >> 20);
}

// Bits [lo, hi] of word q of a mask.
__device__ __forceinline__ uint32_t vox_bits(int32_t lo, int32_t hi, int q) {
    lo = max(lo - 32 * q, 0);
    hi = min(hi - 32 * q, 31);
    return lo > hi ? 0u : (0xFFFFFFFFu << lo) & (0xFFFFFFFFu >> (31 - hi));
}

// The 32 x 32 bit matrix of the lanes' words, transposed.
__device__ __forceinline__ uint32_t vox_transpose(uint32_t x, int lane) {
    const uint32_t masks[5] = {0x0000FFFFu, 0x00FF00FFu, 0x0F0F0F0Fu, 0x33333333u, 0x55555555u};
#pragma unroll
    for (int i = 0; i < 5; ++i) {
        const int s = 16 >> i;
        const uint32_t m = masks[i], y = __shfl_xor_sync(0xFFFFFFFFu, x, s);
        x = lane & s ? (x & ~m) | ((y >> s) & m) : (x & m) | ((y & m) << s);
    }
    return x;
}

// Level 0.  In an 8^3 tile a word holds 4 x 4 columns of 2 layers (voxel bits
// x0 y0 z0 x1 y1), so a warp takes two blocks of 4 x 4 columns beside each
// other in x, a column per lane in bit order (x0 y0 x1 y1, then the block).
// Each lane gathers its column's layers as a mask of NQ words; a transposition
// across the warp then gives lane k the 32 columns' bits of layer 32 q + k, and
// a pair of lanes two layers, of which the even one writes the first block's
// word and the odd one the second's.  Words are written whole: no atomics, and
// no clearing first.  Warps (pi, bj): tile column pi0 + .., block row bj0 + ...
//
// Bound by instruction issue (about 35 a cell and warp, for slabs mostly).  One
// thread per column with a loop over layers and an atomic per word took 920 us
// on 2048 x 16384 cells at (4, 8, 2), against 20 us to read the cells; now 82.
template <int NQ>
__global__ void __launch_bounds__(128)
    k_vox_level0(const WorldDev w, const VoxelDev v, int32_t pi0, int32_t bj0, int32_t npi,
                 int32_t n_warps) {
    const int32_t warp = (int32_t)((blockIdx.x * blockDim.x + threadIdx.x) >> 5);
    if (warp >= n_warps) return;
    const int lane = threadIdx.x & 31;
    const int32_t pi = pi0 + warp % npi, bj = bj0 + warp / npi;
    const int32_t i = pi * 8 + (lane >> 4) * 4 + (lane & 1) + ((lane >> 1) & 2);
    const int32_t j = bj * 4 + ((lane >> 1) & 1) + ((lane >> 2) & 2);
    const int32_t nz = v.nz[0];
    const uint32_t recip = (1u << 20) / (uint32_t)v.vz + 1;
    uint32_t mask[NQ];
#pragma unroll
    for (int q = 0; q < NQ; ++q) mask[q] = 0;
    if (i < v.nx[0] && j < v.ny[0]) {
        int32_t floor_max = 0;
        auto add = [&](uint32_t node) {
            const int32_t h0 = node & 0xFF, h1 = (node >> 8) & 0xFF, h2 = (node >> 16) & 0xFF;
            // floor: layers k with k vz <= h0 (the highest floor's hold all);
            // slab: h1 <= (k+1) vz and k vz <= h2
            floor_max = max(floor_max, h0);
            if (h2 > h0) {  // node form: slab iff top > floor
                const int32_t ka = max(vox_div(h1 + v.vz - 1, recip) - 1, 0);
                const int32_t kb = min(vox_div(h2, recip), nz - 1);
#pragma unroll
                for (int q = 0; q < NQ; ++q) mask[q] |= vox_bits(ka, kb, q);
            }
        };
        const int32_t x0 = i * v.vx, x1 = min(x0 + v.vx, w.W);
        const int32_t y1 = min((j + 1) * v.vy, w.H);
        if (v.vx == 4 && (w.W & 3) == 0 && !w.pair) {  // one 16-byte load a row
            for (int32_t y = j * v.vy; y < y1; ++y) {
                const uint4 c = __ldg(reinterpret_cast<const uint4 *>(
                    w.base + (uint32_t)y * (uint32_t)w.W + (uint32_t)x0));
                add(c.x);
                add(c.y);
                add(c.z);
                add(c.w);
            }
        } else {
            for (int32_t y = j * v.vy; y < y1; ++y)
                for (int32_t x = x0; x < x1; ++x) add(level0_node(w, x, y));
        }
        const int32_t kb = min(vox_div(floor_max, recip), nz - 1);
#pragma unroll
        for (int q = 0; q < NQ; ++q) mask[q] |= vox_bits(0, kb, q);
    }
    auto spread = [](uint32_t b) {  // nibble g of 16 bits to the low half of byte g
        b = (b | (b << 8)) & 0x00FF00FFu;
        return (b | (b << 4)) & 0x0F0F0F0Fu;
    };
    const int32_t tz = (nz + 7) >> 3, tj = bj >> 1;
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
        const uint32_t own = vox_transpose(mask[q], lane);
        const uint32_t other = __shfl_xor_sync(0xFFFFFFFFu, own, 1);
        const uint32_t word = lane & 1 ? spread(other >> 16) | (spread(own >> 16) << 4)
                                       : spread(own & 0xFFFFu) | (spread(other & 0xFFFFu) << 4);
        const int32_t z = 32 * q + (lane & ~1);
        if ((z >> 3) < tz)
            v.words[v.off[0] + (uint32_t)(((z >> 3) * v.ty[0] + tj) * v.tx[0] + pi) * 16 +
                    (((z >> 1) & 1) | ((lane & 1) << 1) | ((bj & 1) << 2) | (((z >> 2) & 1) << 3))] =
                word;
    }
}

// One word of level l >= 1, tile (tx, ty, tz) and word wi = Z1 X2 Y2 Z2 (lowest
// first): its voxels' children fill the eight consecutive words Z1 * 8 .. of
// child tile 2 t + (X2, Y2, Z2), child word c = Z0 X1 Y1, in whose byte X0 Y0
// lie the eight children of one voxel.  So nibble c of the word says which
// bytes of child word c are not zero.
__device__ __forceinline__ void vox_up_word(const VoxelDev &v, int l, int32_t tx, int32_t ty,
                                            int32_t tz, uint32_t wi) {
    const int32_t cx = 2 * tx + ((wi >> 1) & 1), cy = 2 * ty + ((wi >> 2) & 1),
                  cz = 2 * tz + (wi >> 3);
    uint32_t word = 0;
    if (cx < v.tx[l - 1] && cy < v.ty[l - 1] && cz < ((v.nz[l - 1] + 7) >> 3)) {
        // (not the read-only path: the words may be this kernel's own)
        const uint4 *p = reinterpret_cast<const uint4 *>(
            v.words + v.off[l - 1] + (uint32_t)((cz * v.ty[l - 1] + cy) * v.tx[l - 1] + cx) * 16 +
            (wi & 1) * 8);
        const uint4 a = __ldcg(p), b = __ldcg(p + 1);
        const uint32_t c[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const uint32_t any = (((c[k] & 0x7F7F7F7Fu) + 0x7F7F7F7Fu) | c[k]) >> 7 & 0x01010101u;
            word |= ((any * 0x01020408u) >> 24 & 0xFu) << (4 * k);
        }
    }
    v.words[v.off[l] + (uint32_t)((tz * v.ty[l] + ty) * v.tx[l] + tx) * 16 + wi] = word;
}

// The tiles of a level over level-0 columns [i0, i1) x [j0, j1).
struct VoxTiles {
    int32_t x, y, nx, ny, n_words;
};
__host__ __device__ __forceinline__ VoxTiles vox_tiles(const VoxelDev &v, int l, int32_t i0,
                                                       int32_t j0, int32_t i1, int32_t j1) {
    VoxTiles t;
    t.x = i0 >> (l + 3);
    t.y = j0 >> (l + 3);
    t.nx = ((i1 - 1) >> (l + 3)) - t.x + 1;
    t.ny = ((j1 - 1) >> (l + 3)) - t.y + 1;
    t.n_words = t.nx * t.ny * ((v.nz[l] + 7) >> 3) * 16;
    return t;
}

__device__ __forceinline__ void vox_up_index(const VoxelDev &v, int l, const VoxTiles &t, int32_t n) {
    const int32_t tile = n >> 4;
    vox_up_word(v, l, t.x + tile % t.nx, t.y + (tile / t.nx) % t.ny, tile / (t.nx * t.ny),
                (uint32_t)n & 15);
}

__global__ void __launch_bounds__(256) k_vox_up(const VoxelDev v, int l, const VoxTiles t) {
    const int32_t n = (int32_t)(blockIdx.x * blockDim.x + threadIdx.x);
    if (n < t.n_words) vox_up_index(v, l, t, n);
}

// Levels l_from.. of a small region in one block (its own writes are visible to
// it after a barrier).
__global__ void __launch_bounds__(kVoxTailThreads)
    k_vox_tail(const VoxelDev v, int l_from, int32_t i0, int32_t j0, int32_t i1, int32_t j1) {
    for (int l = l_from; l < v.levels; ++l) {
        const VoxTiles t = vox_tiles(v, l, i0, j0, i1, j1);
        for (int32_t n = threadIdx.x; n < t.n_words; n += blockDim.x) vox_up_index(v, l, t, n);
        __syncthreads();
    }
}

// The level to which every ray of a camera at o first descends from the top
// level (one step each level): the first one where the camera's voxel is empty,
// else 0.  Lane k looks at level k.  A voxel's index on level k is the quotient's
// floor there, provided that halving it gives the index of level k + 1 (rounding
// may differ for an extent that is no power of two).  Rays start at o only if the
// camera lies in the box of level 0: above it, it may still lie in the last
// voxels of coarser levels, which reach past it, but its rays start where they
// enter the box, and from the top.  Every lane of the warp calls.
__device__ __forceinline__ int vox_start(const VoxelDev &v, const VoxLevel *lv, const float *o,
                                         const int32_t *vs, const int32_t *ve, int lane) {
    constexpr uint32_t full = 0xFFFFFFFFu;
    const int top = v.levels - 1, k = min(lane, top);
    int32_t n[3];
    bool good = lane <= top;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const float f = floorf(vox_quot(o[a], vs[a], ve[a], k));
        good = good && f >= 0.0f && f < (float)lv[k].n[a];
        n[a] = (int32_t)f;
        const int32_t parent = __shfl_down_sync(full, n[a], 1);
        good = good && (k == top || n[a] >> 1 == parent);
    }
    const bool occ = good && vox_occupied(v, lv[k], (uint32_t)n[0], (uint32_t)n[1], (uint32_t)n[2]);
    const uint32_t goods = __ballot_sync(full, good), occs = __ballot_sync(full, occ);
    if (!(goods & 1)) return top;
    // bit 31 is the top level: the run of occupied voxels from there on
    const int down = min(__clz(~(occs << (31 - top))), top);
    return goods >> (top - down) & 1 ? top - down : min(top - down + 1, top);
}

// One warp traces 8 x 4 pixels, a ray per lane, all lanes step by step together
// (the vote at the head of the loop keeps them so).
//
// On an axis that the ray descends along, voxel index n is held as ~n, so that
// the ray always moves toward larger indices: the first child along it is
// 2 n, and a parent is left where the new index is even.
//
// A step needs the times at which the ray crosses the exit planes of its voxel.
// A plane's coordinate bnd is an integer below 2^24, exact in float, and its
// time is (bnd - o) inv, the same whichever level the plane is met on: so both
// are carried, and a step recomputes those of the axes whose plane changes (an
// advance moves one plane; a climb or a descent those whose child is not the
// last along the ray).  POW2: every extent is a power of two; then the voxel
// that holds p(t) follows from comparing p(t) with the midplane, as the
// quotient that defines it is an exact scaling.
//
// Bound by instruction issue.  12 views of 1280 x 800, (4, 8, 2), 4 samples:
// 2.48 ms, 2.61 ms if every ray descends from the top level, 3.46 ms with rows of
// 32 pixels per warp and every plane made anew each step.
template <bool POW2>
__global__ void __launch_bounds__(kVoxThreads, kVoxMinBlocks)
    k_vox_trace(const RenderParams p, const VoxelDev v, const VoxelParams q) {
    __shared__ VoxLevel s_lv[kVoxMaxLevels];
    __shared__ float s_frac[kVoxFracTable];
    if (threadIdx.x < (unsigned)v.levels) {
        const int l = threadIdx.x;
        s_lv[l] = VoxLevel{v.off[l], v.tx[l], v.ty[l], 0, {v.nx[l], v.ny[l], v.nz[l]}, 0};
    }
    if (threadIdx.x < (unsigned)min(q.inner, kVoxFracTable))
        s_frac[threadIdx.x] = __fdiv_rn(__fadd_rn((float)threadIdx.x, 0.5f), (float)q.inner);
    __syncthreads();
    constexpr uint32_t full = 0xFFFFFFFFu;
    const float inf = __int_as_float(0x7f800000);
    const CamDev &c = p.cams[blockIdx.y];
    const int lane = threadIdx.x & 31;
    const uint32_t tile = blockIdx.x * (kVoxThreads / 32) + (threadIdx.x >> 5);
    const int32_t px = (int32_t)(tile % c.tiles_x) * 8 + (lane & 7);
    const int32_t py = (int32_t)(tile / c.tiles_x) * 4 + (lane >> 3);
    if (py - (lane >> 3) >= (int32_t)c.h) return;  // (no tile of this image: the whole warp)
    const bool inside = px < (int32_t)c.w && py < (int32_t)c.h;
    const int32_t a = 2 * px + 1 - (int32_t)c.w, b = (int32_t)c.h - 1 - 2 * py;
    const float inv_s = 1.0f / 65536.0f;
    const int32_t vs[3] = {v.vx, v.vy, v.vz};
    const int32_t ve[3] = {pow2_log2(v.vx), pow2_log2(v.vy), pow2_log2(v.vz)};
    // o, d: the ray; ot, inv: a plane's time is (plane - ot) inv, infinite on
    // an axis that the ray does not move along
    float o[3], d[3], ot[3], inv[3], box[3];
    int32_t neg[3];  // -1 on a mirrored axis, else 0
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        o[k] = __fmul_rn(__int2float_rn(c.o[k]), inv_s);
        d[k] = __fmul_rn(__int2float_rn(c.F[k] + a * c.R[k] + b * c.U[k]), inv_s);
        neg[k] = d[k] < 0.0f ? -1 : 0;
    }
    box[0] = (float)(v.nx[0] * v.vx);
    box[1] = (float)(v.ny[0] * v.vy);
    box[2] = (float)(v.nz[0] * v.vz);
    const float dl = __fsqrt_rn(__fadd_rn(__fadd_rn(__fmul_rn(d[0], d[0]), __fmul_rn(d[1], d[1])),
                                          __fmul_rn(d[2], d[2])));
    float t0 = 0.0f, t1 = __fdiv_rn(q.far_dist, dl);
    bool miss = !inside;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        if (d[k] != 0.0f) {
            ot[k] = o[k];
            inv[k] = __fdiv_rn(1.0f, d[k]);
            const float ta = __fmul_rn(__fsub_rn(0.0f, o[k]), inv[k]);
            const float tb = __fmul_rn(__fsub_rn(box[k], o[k]), inv[k]);
            t0 = fmaxf(t0, fminf(ta, tb));
            t1 = fminf(t1, fmaxf(ta, tb));
        } else {
            ot[k] = -inf;
            inv[k] = 1.0f;
            if (o[k] < 0.0f || o[k] > box[k]) miss = true;
        }
    }
    uint32_t cell = 0xFFFFFFFFu;
    uint8_t layer = 255;
    float depth = inf;
    const int top = v.levels - 1;
    int l = vox_start(v, s_lv, o, vs, ve, lane);
    float scale = __int_as_float((127 + l) << 23);  // 2^l
    float t = t0;
    int ent = -1;
    int32_t idx[3];                // mirrored
    float size[3], bnd[3], tk[3];  // extent along the ray at level 0; exit plane; its time
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const float pk = __fadd_rn(o[k], __fmul_rn(d[k], t));
        const float cf = floorf(vox_quot(pk, vs[k], ve[k], l));
        const int32_t n = (int32_t)fminf(fmaxf(cf, 0.0f), (float)(s_lv[l].n[k] - 1));
        idx[k] = n ^ neg[k];
        size[k] = neg[k] ? -(float)vs[k] : (float)vs[k];
        bnd[k] = (float)((n + 1 + neg[k]) * (vs[k] << l));
        tk[k] = __fmul_rn(__fsub_rn(bnd[k], ot[k]), inv[k]);
    }
    bool run = !miss && t0 < t1;
    for (int step = top - l; step < q.outer && __any_sync(full, run); ++step) {
        if (!run) continue;
        const float t_out = fminf(fminf(tk[0], tk[1]), tk[2]);
        const VoxLevel &lv = s_lv[l];
        const uint32_t x = (uint32_t)(idx[0] ^ neg[0]), y = (uint32_t)(idx[1] ^ neg[1]),
                       z = (uint32_t)(idx[2] ^ neg[2]);
        // a child past the level's end (the last parent of an odd count) is empty
        const bool occ = (x < (uint32_t)lv.n[0]) & (y < (uint32_t)lv.n[1]) &
                         (z < (uint32_t)lv.n[2]) && vox_occupied(v, lv, x, y, z);
        if (occ && l > 0) {
            --l;
            scale *= 0.5f;
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                // the first child along the ray on the axis last crossed,
                // else the one that holds p(t)
                const float mid = fmaf(-scale, size[k], bnd[k]);  // midplane
                const float pk = __fadd_rn(o[k], __fmul_rn(d[k], t));
                bool upper;
                if (POW2) upper = pk >= mid;
                else upper = vox_quot(pk, vs[k], ve[k], l) >= (float)(2 * (idx[k] ^ neg[k]) + 1);
                const bool last = k != ent && upper != (neg[k] != 0);
                idx[k] = 2 * idx[k] + (last ? 1 : 0);
                if (!last) {
                    bnd[k] = mid;
                    tk[k] = __fmul_rn(__fsub_rn(mid, ot[k]), inv[k]);
                }
            }
            continue;
        }
        if (occ) {
            const float span = __fsub_rn(fminf(t_out, t1), t);
            bool found = false;
            for (int s = 0; s < q.inner && !found; ++s) {
                const float frac = s < kVoxFracTable
                                       ? s_frac[s]
                                       : __fdiv_rn(__fadd_rn((float)s, 0.5f), (float)q.inner);
                const float ts = __fadd_rn(t, __fmul_rn(span, frac));
                const float sx = __fadd_rn(o[0], __fmul_rn(d[0], ts));
                const float sy = __fadd_rn(o[1], __fmul_rn(d[1], ts));
                const float sz = __fadd_rn(o[2], __fmul_rn(d[2], ts));
                const float fx = floorf(sx), fy = floorf(sy);
                if (!(fx >= 0.0f && fx < (float)p.world.W && fy >= 0.0f && fy < (float)p.world.H))
                    continue;
                const uint32_t node = level0_node(p.world, (int32_t)fx, (int32_t)fy);
                const float h0 = (float)(node & 0xFF), h1 = (float)((node >> 8) & 0xFF),
                            h2 = (float)((node >> 16) & 0xFF);
                const bool fl = sz <= h0;
                const bool up = h2 > h0 && sz >= h1 && sz <= h2;
                if (fl || up) {
                    found = true;
                    cell = (uint32_t)fy * (uint32_t)p.world.W + (uint32_t)fx;
                    layer = fl ? 0 : 1;
                    depth = __fmul_rn(ts, dl);
                }
            }
            if (found) run = false;
        }
        if (t_out >= t1) run = false;
        if (!run) continue;
        ent = tk[0] == t_out ? 0 : (tk[1] == t_out ? 1 : 2);
        t = t_out;
        const int32_t ni = (ent == 0 ? idx[0] : ent == 1 ? idx[1] : idx[2]) + 1;
        const int32_t nn = ent == 0 ? neg[0] : ent == 1 ? neg[1] : neg[2];
        if ((uint32_t)(ni ^ nn) >= (uint32_t)lv.n[ent]) {
            run = false;
            continue;
        }
        const int32_t climb = (l < v.levels - 1 ? 1 : 0) & ~ni;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            if (k == ent) {
                idx[k] = ni;
                bnd[k] = fmaf(scale, size[k], bnd[k]);
            }
            // the parent's exit plane, where this child is its first along the ray
            const bool first = climb & ~idx[k] & 1;
            if (first) bnd[k] = fmaf(scale, size[k], bnd[k]);
            if (first || k == ent) tk[k] = __fmul_rn(__fsub_rn(bnd[k], ot[k]), inv[k]);
            idx[k] >>= climb & 1;
        }
        if (climb & 1) {
            ++l;
            scale *= 2.0f;
        }
    }
    if (!inside) return;
    const uint32_t pix = (uint32_t)py * c.w + (uint32_t)px;
    if (c.hit_cell) c.hit_cell[pix] = cell;
    if (c.layer) c.layer[pix] = layer;
    if (c.depth) c.depth[pix] = depth;
}

}  // namespace

int voxel_repair(const WorldDev &w, const VoxelDev &v, int32_t x0, int32_t y0, int32_t x1,
                 int32_t y1, void *stream) {
    cudaStream_t s = (cudaStream_t)stream;
    if (x1 <= x0 || y1 <= y0) return 0;
    const int32_t i0 = x0 / v.vx, i1 = (x1 - 1) / v.vx + 1, j0 = y0 / v.vy, j1 = (y1 - 1) / v.vy + 1;
    {
        const int32_t pi0 = i0 >> 3, npi = ((i1 - 1) >> 3) - pi0 + 1;
        // block rows in pairs at the grid's end: a tile's rows past it are written too
        const int32_t bj0 = j0 >> 2, bj1 = j1 == v.ny[0] ? 2 * v.ty[0] : ((j1 - 1) >> 2) + 1;
        const int32_t n = npi * (bj1 - bj0), blocks = (n + 3) / 4;
        const int nq = (v.nz[0] + 31) / 32;
        if (nq > 4) k_vox_level0<8><<<blocks, 128, 0, s>>>(w, v, pi0, bj0, npi, n);
        else if (nq > 2) k_vox_level0<4><<<blocks, 128, 0, s>>>(w, v, pi0, bj0, npi, n);
        else k_vox_level0<2><<<blocks, 128, 0, s>>>(w, v, pi0, bj0, npi, n);
    }
    int l = 1;
    for (; l < v.levels; ++l) {
        const VoxTiles t = vox_tiles(v, l, i0, j0, i1, j1);
        if (t.n_words <= kVoxTailWords) break;
        k_vox_up<<<(t.n_words + 255) / 256, 256, 0, s>>>(v, l, t);
    }
    if (l < v.levels) k_vox_tail<<<1, kVoxTailThreads, 0, s>>>(v, l, i0, j0, i1, j1);
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

int launch_voxel_trace(const RenderParams &p, const VoxelDev &v, const VoxelParams &q,
                       uint32_t n_cams, uint32_t max_tiles, void *stream) {
    const uint32_t per = kVoxThreads / 32;
    const dim3 grid((max_tiles + per - 1) / per, n_cams);
    const bool pow2 = pow2_log2(v.vx) >= 0 && pow2_log2(v.vy) >= 0 && pow2_log2(v.vz) >= 0;
    if (pow2) k_vox_trace<true><<<grid, kVoxThreads, 0, (cudaStream_t)stream>>>(p, v, q);
    else k_vox_trace<false><<<grid, kVoxThreads, 0, (cudaStream_t)stream>>>(p, v, q);
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

}  // namespace hf
