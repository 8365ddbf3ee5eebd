// hf_single.cu -- the trace kernels that follow each ray by itself: renders with a
// step limit of the caller's or with fetch counters, and views whose rays lie too
// far apart for beams (beams_fit in hf_rules.h).
//
// One warp owns one tile of tile_w x tile_h pixels; each lane traces the tile's
// pixels lane, lane + 32, ... by hierarchical DDA over the min/max pyramid
// (cast_single in hf_cast.h): every branch is decided with exact integer
// arithmetic on 32-bit operands and 64-bit products (times are rationals num/den
// with 0 <= num <= 2^30 and 0 < den < 2^21), so hit cell, layer and face equal the
// definition bit for bit.
//
// Bound by instruction issue.  Lanes go on to their shadow rays while others
// still follow their primary rays.  In the form that beams need (passes of the
// whole warp, blocks of 128 threads) these kernels took 2 % longer on the average
// of 626 calls (views of 64 x 48 to 1920 x 1080 over four worlds), batches of small
// views 6 %.
#include <cuda_runtime.h>
#include <math.h>

#include "hf_trace.h"

namespace hf {
namespace {

constexpr int kSingleThreads = trace_threads(kTraceGeneral);
// Resident blocks per SM asked of the register allocator (<= 85 registers; four
// blocks, 64 registers: 3 % slower over the same calls).
constexpr int kSingleMinBlocks = 3;

__device__ __forceinline__ uint32_t load_word(const WorldDev &w, int level, int32_t x, int32_t y) {
    return __ldg(w.base + w.off[level] + (uint32_t)y * w.stride[level] + (uint32_t)x);
}

// Node-form word of level-0 cell (x, y) for the storage the kernel was
// instantiated for (the choice is made at compile time).
template <bool PAIR>
__device__ __forceinline__ uint32_t level0_word(const WorldDev &w, int32_t x, int32_t y) {
    if (PAIR)
        return pair_node(__ldg(w.base + (uint32_t)y * ((uint32_t)w.W >> 1) + ((uint32_t)x >> 1)),
                         (uint32_t)x & 1);
    return load_word(w, 0, x, y);
}

// The cosine of a face with the sun's direction (by a switch: as selects, it cost
// renders with shadows 2 %, by their registers).
__device__ __forceinline__ float face_cosine(uint8_t face, const float *ln) {
    switch (face) {
        case kFaceNX: return -ln[0];
        case kFacePX: return ln[0];
        case kFaceNY: return -ln[1];
        case kFacePY: return ln[1];
        case kFaceNZ: return -ln[2];
        case kFacePZ: return ln[2];
        default: return 0.0f;
    }
}

// Writes one pixel's outputs.
__device__ __forceinline__ void store_pixel(const RenderParams &p, const CamDev &c, uint32_t pix,
                                            const Hit &ph, float depth, bool visible,
                                            bool shadows) {
    const bool hit = ph.face < kFaceError;
    if (shadows && c.shadow) __stcs(c.shadow + pix, (uint8_t)(visible ? 0 : 1));
    if (c.hit_cell)
        __stcs(c.hit_cell + pix,
               hit ? (uint32_t)ph.cy * (uint32_t)p.world.W + (uint32_t)ph.cx : 0xFFFFFFFFu);
    if (c.layer) __stcs(c.layer + pix, hit ? ph.layer : (uint8_t)255);
    if (c.face) __stcs(c.face + pix, ph.face);
    if (c.depth) __stcs(c.depth + pix, depth);
    if (c.rgba)
        __stcs(c.rgba + pix,
               hit ? shade(ph.word >> 24 & 7, face_cosine(ph.face, p.sun_n), visible) : kSky);
}

// One pixel: its primary ray, then (with shadows) the shadow ray, which
// reuses the same traversal loop and registers.
template <bool SHADOWS, bool STATS, bool PAIR>
__device__ __forceinline__ void trace_pixel(const RenderParams &p, const LevelDev *lvt,
                                            const CamDev &c, int start,
                                            int32_t px, int32_t py, Counters &cnt,
                                            Counters &scnt, uint32_t &nshadow, bool &err) {
    Ray r = primary_ray(c, px, py);
    Hit ph;  // primary hit, kept while the shadow ray runs
    float depth = __int_as_float(0x7f800000);
    bool visible = true;
    bool shadow_pass = false;
    for (;;) {
        Hit h;
        // one call site: lanes in the primary and in the shadow pass run the
        // same traversal code together
        const bool sp = SHADOWS && shadow_pass;
        Counters pc{0, 0};
        cast_single<STATS, PAIR, SHADOWS, false>(
            p.world.W, p.world.H, p.world.base, lvt, r, sp ? min(kShadowStart, p.shadow_mip) : start,
            sp ? p.shadow_mip : p.mip_start, p.max_steps, nullptr, h, pc);
        if (STATS) {
            Counters &dst = sp ? scnt : cnt;
            dst.nodes += pc.nodes;
            dst.cells += pc.cells;
        }
        if (h.face == kFaceError) err = true;
        if (SHADOWS && shadow_pass) {
            visible = h.face == kFaceMiss;
            break;
        }
        ph = h;
        const bool hit = h.face < kFaceError;
        if (hit) {
            const float fx = (float)r.dx, fy = (float)r.dy, fz = (float)r.dz;
            depth = ((float)h.tnum / (float)h.tden) * sqrtf(fx * fx + fy * fy + fz * fz) *
                    (1.0f / 65536.0f);
        }
        if (!SHADOWS || !hit) break;
        if (h.face == kFaceInside) {
            visible = false;
            break;
        }
        // shadow ray: floor of the hit point, one unit outward along the face normal
        const float rcp_t = 1.0f / (float)h.tden;
        int32_t sxp = r.ox + floor_div_small((int64_t)h.tnum * r.dx, h.tden, rcp_t);
        int32_t syp = r.oy + floor_div_small((int64_t)h.tnum * r.dy, h.tden, rcp_t);
        int32_t szp = r.oz + floor_div_small((int64_t)h.tnum * r.dz, h.tden, rcp_t);
        switch (h.face) {
            case kFaceNX: sxp -= 1; break;
            case kFacePX: sxp += 1; break;
            case kFaceNY: syp -= 1; break;
            case kFacePY: syp += 1; break;
            case kFaceNZ: szp -= 1; break;
            default: szp += 1; break;
        }
        if (STATS) nshadow++;
        if (p.sun_bounds) {
            // the start cell's proven bounds decide most shadow rays at once:
            // at or below F occluded, at or above G lit (hf_sun.cu)
            int32_t bx = sxp >> kShift, by = syp >> kShift;
            if (p.sun[0] < 0 && (sxp & 0xFFFF) == 0) bx -= 1;
            if (p.sun[1] < 0 && (syp & 0xFFFF) == 0) by -= 1;
            if ((uint32_t)bx < (uint32_t)p.world.W && (uint32_t)by < (uint32_t)p.world.H) {
                const uint32_t fg = __ldg(p.sun_bounds + (uint32_t)by * (uint32_t)p.world.W + (uint32_t)bx);
                if (STATS) scnt.cells++;
                if (szp <= (int32_t)((fg & 0xFFFFu) << 8)) {
                    visible = false;
                    break;
                }
                if (szp >= (int32_t)((fg >> 16) << 8)) break;
            }
        }
        r.ox = sxp;
        r.oy = syp;
        r.oz = szp;
        r.dx = p.sun[0];
        r.dy = p.sun[1];
        r.dz = p.sun[2];
        shadow_pass = true;
    }
    store_pixel(p, c, (uint32_t)py * c.w + (uint32_t)px, ph, depth, visible, SHADOWS);
}

// Start level of a camera's primary rays: the largest level l <= mip_start
// whose node around the camera cell has every top below the camera, but not
// below level min(2, mip_start) (a measured floor: climbing out of levels 0
// and 1 costs more steps than the two descents it saves).  Node tops only
// grow with the level, so the levels under the camera are 0..l; lane k tests
// level k.  A camera outside the grid starts at mip_start.  The traversal is
// exact from any start level (a ray climbs as it crosses parent boundaries);
// the rule only saves descents through nodes around the camera that cannot
// be empty.
template <bool PAIR>
__device__ __forceinline__ int primary_start(const RenderParams &p, const CamDev &c, int lane) {
    const WorldDev &w = p.world;
    const int32_t cx = c.o[0] >> kShift, cy = c.o[1] >> kShift;
    if ((uint32_t)cx >= (uint32_t)w.W || (uint32_t)cy >= (uint32_t)w.H) return p.mip_start;
    bool above = false;
    if (lane <= p.mip_start) {
        const uint32_t word =
            lane ? load_word(w, lane, cx >> lane, cy >> lane) : level0_word<PAIR>(w, cx, cy);
        const int32_t top = (word >> 16) & 0xFF;  // every level in node form
        above = c.o[2] > (top << kShift);
    }
    const uint32_t mask = __ballot_sync(0xFFFFFFFFu, above);
    return max(min(2, p.mip_start), __ffs(~mask) - 2);
}

// One warp renders one tile: lane l traces the tile's pixels l, l+32, ...
template <bool SHADOWS, bool STATS, bool PAIR>
__device__ __forceinline__ void trace_tile(const RenderParams &p, const LevelDev *lvt,
                                           const CamDev &c, uint32_t local_tile, int lane) {
    const uint32_t tx = local_tile % c.tiles_x, ty = local_tile / c.tiles_x;
    const int32_t tw_log2 = p.tile_w_log2;
    const int32_t x0 = (int32_t)tx << tw_log2, y0 = (int32_t)ty << p.tile_h_log2;
    const int32_t npix = 1 << (tw_log2 + p.tile_h_log2);
    Counters cnt{0, 0}, scnt{0, 0};
    uint32_t nshadow = 0, nrays = 0;
    bool err = false;
    const int start = primary_start<PAIR>(p, c, lane);
    for (int i = lane; i < npix; i += 32) {
        const int32_t px = x0 + (i & ((1 << tw_log2) - 1));
        const int32_t py = y0 + (i >> tw_log2);
        if (px < (int32_t)c.w && py < (int32_t)c.h) {
            trace_pixel<SHADOWS, STATS, PAIR>(p, lvt, c, start, px, py, cnt, scnt, nshadow, err);
            if (STATS) nrays++;
        }
    }
    if (__any_sync(0xFFFFFFFFu, err) && lane == 0) atomicOr(p.status, 1u);
    if (STATS) {
        const uint32_t vn = __reduce_add_sync(0xFFFFFFFFu, cnt.nodes);
        const uint32_t vc = __reduce_add_sync(0xFFFFFFFFu, cnt.cells);
        const uint32_t vr = __reduce_add_sync(0xFFFFFFFFu, nrays);
        const uint32_t vs = __reduce_add_sync(0xFFFFFFFFu, nshadow);
        const uint32_t vf = __reduce_add_sync(0xFFFFFFFFu, scnt.nodes + scnt.cells);
        if (lane == 0) {
            atomicAdd(p.stats + 0, (unsigned long long)vn);
            atomicAdd(p.stats + 1, (unsigned long long)vc);
            atomicAdd(p.stats + 2, (unsigned long long)vr);
            atomicAdd(p.stats + 3, (unsigned long long)vs);
            atomicAdd(p.stats + 4, (unsigned long long)vf);
        }
    }
}

// Copy camera i into this warp's shared slot (fields are then read on demand
// instead of being held in registers for the whole tile).
__device__ __forceinline__ const CamDev &stage_cam(CamDev *slot, const CamDev *cams, uint32_t i,
                                                   int lane) {
    static_assert(sizeof(CamDev) % 4 == 0 && sizeof(CamDev) / 4 <= 32, "one word per lane");
    const uint32_t *src = reinterpret_cast<const uint32_t *>(cams + i);
    uint32_t *dst = reinterpret_cast<uint32_t *>(slot);
    __syncwarp();
    if (lane < (int)(sizeof(CamDev) / 4)) dst[lane] = src[lane];
    __syncwarp();
    return *slot;
}

// Persistent batched kernel: warps pop (camera, tile) items from one atomic
// counter until the batch is drained.  One launch renders every camera.
template <bool SHADOWS, bool STATS, bool PAIR>
__global__ void __launch_bounds__(kSingleThreads, kSingleMinBlocks) k_single_batched(const RenderParams p) {
    __shared__ uint32_t s_base[kMaxCams + 1];
    __shared__ CamDev s_cam[kSingleThreads / 32];
    __shared__ LevelDev s_lv[kMaxLevels + 1];
    const uint32_t n = p.hdr->n_cams;
    const uint32_t total = p.hdr->total_tiles;
    prefetch_world(p);
    for (uint32_t i = threadIdx.x; i < n; i += blockDim.x) s_base[i] = p.cams[i].tile_base;
    fill_levels(s_lv, p.world);
    __syncthreads();
    const int lane = threadIdx.x & 31;
    for (;;) {
        uint32_t t = 0;
        if (lane == 0) t = atomicAdd(&p.hdr->counter, 1u);
        t = __shfl_sync(0xFFFFFFFFu, t, 0);
        if (t >= total) break;
        // last camera whose first tile is <= t
        uint32_t lo = 0, hi = n;
        while (hi - lo > 1) {
            const uint32_t mid = (lo + hi) >> 1;
            if (s_base[mid] <= t) lo = mid;
            else hi = mid;
        }
        const CamDev &c = stage_cam(&s_cam[threadIdx.x >> 5], p.cams, lo, lane);
        trace_tile<SHADOWS, STATS, PAIR>(p, s_lv, c, t - s_base[lo], lane);
    }
}

// Plain kernel: one camera, one warp per tile, grid covers the image once.
// The camera record is a kernel parameter, so a plain render needs no copy of
// it to the device; each warp stages it in shared memory like the batched
// kernel (reading the fields from parameter space instead changes the
// traversal's register allocation, measured 3-8 % slower on large images).
template <bool SHADOWS, bool STATS, bool PAIR>
__global__ void __launch_bounds__(kSingleThreads, kSingleMinBlocks)
    k_single_plain(const __grid_constant__ RenderParams p, const __grid_constant__ CamDev cam,
                  uint32_t n_tiles) {
    __shared__ LevelDev s_lv[kMaxLevels + 1];
    __shared__ CamDev s_cam[kSingleThreads / 32];
    prefetch_world(p);
    fill_levels(s_lv, p.world);
    __syncthreads();
    const uint32_t t = blockIdx.x * (kSingleThreads / 32) + (threadIdx.x >> 5);
    if (t >= n_tiles) return;
    const int lane = threadIdx.x & 31;
    const CamDev &c = stage_cam(&s_cam[threadIdx.x >> 5], &cam, 0, lane);
    trace_tile<SHADOWS, STATS, PAIR>(p, s_lv, c, t, lane);
}

template <bool SH, bool ST, bool PA>
const void *batched_ptr() {
    return reinterpret_cast<const void *>(&k_single_batched<SH, ST, PA>);
}

template <bool PA>
const void *batched_fn(bool shadows, bool stats) {
    if (shadows) return stats ? batched_ptr<true, true, PA>() : batched_ptr<true, false, PA>();
    return stats ? batched_ptr<false, true, PA>() : batched_ptr<false, false, PA>();
}

template <bool SH, bool ST, bool PA>
void plain_launch(const RenderParams &p, uint32_t blocks, cudaStream_t s, const CamDev &cam,
                  uint32_t n_tiles) {
    k_single_plain<SH, ST, PA><<<blocks, kSingleThreads, 0, s>>>(p, cam, n_tiles);
}

}  // namespace

const void *single_batched_fn(bool shadows, bool stats, bool pair) {
    return pair ? batched_fn<true>(shadows, stats) : batched_fn<false>(shadows, stats);
}

int launch_single_plain(const RenderParams &p, bool shadows, bool stats, const CamDev &cam,
                       uint32_t n_tiles, void *stream) {
    if (n_tiles == 0) return 0;
    cudaStream_t s = (cudaStream_t)stream;
    const uint32_t warps = kSingleThreads / 32;
    const uint32_t blocks = (n_tiles + warps - 1) / warps;
    using Fn = void (*)(const RenderParams &, uint32_t, cudaStream_t, const CamDev &, uint32_t);
    static const Fn table[8] = {
        plain_launch<false, false, false>, plain_launch<false, false, true>,
        plain_launch<false, true, false>,  plain_launch<false, true, true>,
        plain_launch<true, false, false>,  plain_launch<true, false, true>,
        plain_launch<true, true, false>,   plain_launch<true, true, true>};
    table[(shadows ? 4 : 0) + (stats ? 2 : 0) + (p.world.pair ? 1 : 0)](p, blocks, s, cam, n_tiles);
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

}  // namespace hf

