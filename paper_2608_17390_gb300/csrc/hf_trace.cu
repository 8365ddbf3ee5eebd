// hf_trace.cu -- per-pixel exact ray casting through a two-interval height field, a
// warp's rays together; the allocation-free render.
//
// One warp owns one tile of tile_w x tile_h pixels; lane l takes the tile's
// pixels l, l + 32, ...  The hit cell, layer and face of every ray equal the
// definition bit for bit:
//
//   * ray generation: d = F + (2px+1-w) R + (h-1-2py) U (int32, bounded < 2^21);
//   * the 32 rays of a warp are cast together, in beams (cast_beams): floats
//     with error bounds prove space empty (the hierarchy may only skip
//     known-empty space, Section 3.2 of the paper), and what they leave open is
//     decided in exact integer arithmetic (hf_cast.h): the SOLID predicate of
//     Section 3.1, closed ends, floor unbounded below;
//   * renders with a step limit of the caller's, or with fetch counters, or whose
//     rays lie far apart, follow each ray by itself (hf_single.cu);
//   * a shadow ray starts at the floor of the hit point (an exact floor
//     division: a float estimate and one integer correction), one fixed-point
//     unit outward along the face normal.
#include <cuda_runtime.h>
#include <math.h>

#include <cstring>
#include <mutex>

#include "hf.h"
#include "hf_beam.h"
#include "hf_internal.h"
#include "hf_rules.h"
#include "hf_trace.h"

namespace hf {
namespace {

// Resident 128-thread blocks per SM asked of the register allocator: six leave
// each thread 80 registers (the batched kernel with shadows uses 78, the others
// 72 at most, so that seven fit).  64 views with shadows / 100 frames of 1080p
// without: four blocks 10.62 ms / -, five 9.66 / -, six 9.39 / 8.15, seven (up to
// 4 % more instructions) 9.43 / 8.57.
constexpr int kTraceMinBlocks = 6;
constexpr int kThreads = trace_threads(kTraceBeams);

// Casts one ray per active lane; every lane of the warp calls.  single: each by
// itself; only: of a hit nothing matters but that there is one.
//
// The rays that go the same way and start side by side form a beam (hf_beam.h);
// they are walked, all together, through the runs of columns that it does not
// prove empty, until they have hit or left.  One ray at a time, the same empty
// space costs every lane 15 to 25 dependent node visits; here it costs the warp
// one or two rounds.
//
// Bound by instruction issue, as the traversal of single rays was: 2048 x 2048
// grid with caves and walls, 64 views of 188 M rays with shadows 13.47 -> 9.27
// ms, a 1080p eye-level view with shadows 192 -> 120 us, a hundred 1080p frames
// over 2048 x 16384 cells 17.3 -> 8.0 ms.
template <bool PAIR>
__device__ __forceinline__ void cast_beams(const RenderParams &p, const LevelDev *lvt,
                                           const BeamDir &d, BeamRay q, int32_t oz, int32_t dz,
                                           bool active, bool single, int mip, bool only, Hit &h) {
    BeamHit b;
    b.kind = -1;
    const uint32_t W = (uint32_t)p.world.W, H = (uint32_t)p.world.H;
    const uint32_t *cells = p.world.base;
    const int lane = threadIdx.x & 31;
    // rays that no beam takes: vertical ones, a wide view's, and (below) through corners
    bool alone = active && (single || d.du == 0);
    active = active && !alone && (uint32_t)(d.key & 2 ? ~q.fu : q.fu) < (d.key & 4 ? W : H) &&
             (uint32_t)(d.key & 1 ? ~q.fv : q.fv) < (d.key & 4 ? H : W);
    uint32_t todo = __ballot_sync(kFull, active);
    while (todo) {
        // the first ray left, and the rays that go its way beside it
        const int lead = __ffs(todo) - 1;
        BeamScan s;
        s.key = __reduce_max_sync(kFull, lane == lead ? d.key : -1);
        s.m.u0 = __reduce_max_sync(kFull, lane == lead ? q.fu : (int)0x80000000);
        s.m.v0 = __reduce_max_sync(kFull, lane == lead ? q.fv : (int)0x80000000);
        beam_place(q, s.m);
        bool alive = (todo >> lane & 1) && d.key == s.key &&
                     fabsf(q.pv - d.rho * q.pu) <= kBeamSpread;
        todo &= ~__ballot_sync(kFull, alive);
        s.m.u0 = __reduce_min_sync(kFull, alive ? q.fu : 0x7FFFFFFF);
        beam_place(q, s.m);
        beam_scan(s, p.world, lvt, mip);
        const BeamGrid g = beam_grid(cells, s.m, s.key, W, H);
        int32_t b0, b1;
        while (beam_next<PAIR>(s, lvt, d, q, alive, b0, b1)) {
            const int32_t x1 = b1 - s.m.u0;
            int32_t x = b0 - s.m.u0;
            BeamWalk w;
            if (!beam_enter(d, q, s.m, x, x1, w) && alive) {
                alone = true;
                alive = false;
            }
            // column by column, all rays together
            do {
                if (alive && s.m.u0 + x >= q.fu) {
                    BeamColumn c;
                    const int at = beam_step<PAIR>(g, d, q, s.m, w, x, c);
                    if (at == kBeamOpen) {
                        alive = !beam_settle(g, oz, dz, d, q, s.m, w, x, c, b);
                    } else if (at != kBeamGoing) {
                        alive = false;
                        alone = at == kBeamCorner;
                    }
                    w.row = c.row;
                    w.zl = c.zl;
                }
            } while (__any_sync(kFull, alive) && ++x < x1);
            if (!__any_sync(kFull, alive)) break;
        }
    }
    h.face = kFaceMiss;
    h.layer = 255;
    if (alone) {
        Counters none{0, 0};
        const int level = min(kBeamLevel, mip);
        cast_general<false, PAIR>(lvt, beam_unray(d, q, oz, dz), level, mip, p.max_steps, h, none,
                                  p.status);
    } else if (only) {
        h.face = b.kind < 0 ? kFaceMiss : kFaceInside;
    } else if (b.kind >= 0) {
        h = beam_hit(b, oz, dz, d, q);
    }
}

// The cosine of a face with the sun's direction ln: the normal's axis is face / 2,
// its sign face's lowest bit.
__device__ __forceinline__ float face_cosine(uint8_t face, const float *ln) {
    const float n = face < kFaceNY ? ln[0] : face < kFaceNZ ? ln[1] : ln[2];
    return face == kFaceInside ? 0.0f : face & 1 ? n : -n;
}

// What a warp works on, in shared memory: its camera's record and its tile's
// first pixel.  Fields are read when they are needed instead of being held in
// registers through a cast, where registers decide how many warps fit.
struct TileDev {
    CamDev cam;
    int32_t x0, y0;
};

// Pixel i of the warp's tile.
__device__ __forceinline__ void tile_pixel(const RenderParams &p, const TileDev &t, int i,
                                           int32_t &px, int32_t &py) {
    px = t.x0 + (i & ((1 << p.tile_w_log2) - 1));
    py = t.y0 + (i >> p.tile_w_log2);
}

// One pixel per lane: its primary ray, then (with shadows) the shadow ray, in
// a second pass of the same traversal code.  Every lane of the warp calls.
// WIDE: the view may be a wide one (a launch of one view is not).
template <bool SHADOWS, bool PAIR, bool WIDE>
__device__ __forceinline__ void trace_pixels(const RenderParams &p, const LevelDev *lvt,
                                             const TileDev &t, int i, const BeamDir &sun) {
    const CamDev &c = t.cam;
    int32_t px, py;
    tile_pixel(p, t, i, px, py);
    bool inside = px < (int32_t)c.w && py < (int32_t)c.h;
    Ray r = primary_ray(c, px, py);
    uint32_t tag = kFaceMiss;  // of the primary hit: face and material (bits 8..10)
    bool visible = true;
    bool cast = inside;  // this lane's ray of the pass
#pragma unroll 1
    for (int pass = 0;; ++pass) {
        const bool sp = SHADOWS && pass;
        Hit h;
        const BeamDir d = sp ? sun : beam_dir(r.dx, r.dy, r.dz);
        cast_beams<PAIR>(p, lvt, d, beam_ray(d, r), r.oz, r.dz, cast, WIDE && c.single,
                         sp ? p.shadow_mip : p.mip_start, sp, h);
        if (sp) {
            if (cast) visible = h.face == kFaceMiss;
            break;
        }
        cast = false;
        const bool hit = h.face < kFaceError;
        // the ray again, from the camera: it need not be held through the cast
        if (SHADOWS) {
            asm volatile("" : "+r"(i)::"memory");
            tile_pixel(p, t, i, px, py);
            inside = px < (int32_t)c.w && py < (int32_t)c.h;
        } else {
            asm volatile("" : "+r"(px), "+r"(py)::"memory");
        }
        r = primary_ray(c, px, py);
        const uint32_t pix = (uint32_t)py * c.w + (uint32_t)px;
        if (inside) {
            const uint8_t face = h.face;
            tag = face | (h.word >> 16 & 0x700);
            float depth = __int_as_float(0x7f800000);
            if (hit) {
                const float fx = (float)r.dx, fy = (float)r.dy, fz = (float)r.dz;
                depth = ((float)h.tnum / (float)h.tden) * sqrtf(fx * fx + fy * fy + fz * fz) *
                        (1.0f / 65536.0f);
            }
            if (c.hit_cell)
                __stcs(c.hit_cell + pix, hit ? (uint32_t)h.cy * (uint32_t)p.world.W + (uint32_t)h.cx
                                             : 0xFFFFFFFFu);
            if (c.layer) __stcs(c.layer + pix, hit ? h.layer : (uint8_t)255);
            if (c.face) __stcs(c.face + pix, face);
            if (c.depth) __stcs(c.depth + pix, depth);
        }
        if (!SHADOWS) break;
        if (inside && h.face == kFaceInside) {
            visible = false;
        } else if (inside && hit) {
            // shadow ray: floor of the hit point, one unit outward along the
            // face normal.  The coordinate along the normal is exact: the ray
            // crosses that axis by tnum (its |d| is tden); the other two are
            // floored quotients.
            const bool on_x = h.face <= kFacePX, on_z = h.face >= kFaceNZ;
            const int32_t dn = on_x ? r.dx : on_z ? r.dz : r.dy;
            const int32_t da = on_x ? r.dy : r.dx, db = on_z ? r.dy : r.dz;
            const int32_t qn = dn < 0 ? 1 - h.tnum : h.tnum - 1;  // one unit back
            const float rcp_t = __fdividef(1.0f, (float)h.tden);
            const int32_t qa = floor_div_small((int64_t)h.tnum * da, h.tden, rcp_t);
            const int32_t qb = floor_div_small((int64_t)h.tnum * db, h.tden, rcp_t);
            const int32_t sxp = r.ox + (on_x ? qn : qa);
            const int32_t syp = r.oy + (on_x ? qa : on_z ? qb : qn);
            const int32_t szp = r.oz + (on_z ? qn : qb);
            cast = true;
            if (p.sun_bounds) {
                // the start cell's proven bounds decide most shadow rays at once:
                // at or below F occluded, at or above G lit (hf_sun.cu)
                int32_t bx = sxp >> kShift, by = syp >> kShift;
                if (p.sun[0] < 0 && (sxp & 0xFFFF) == 0) bx -= 1;
                if (p.sun[1] < 0 && (syp & 0xFFFF) == 0) by -= 1;
                if ((uint32_t)bx < (uint32_t)p.world.W && (uint32_t)by < (uint32_t)p.world.H) {
                    const uint32_t fg =
                        __ldg(p.sun_bounds + (uint32_t)by * (uint32_t)p.world.W + (uint32_t)bx);
                    if (szp <= (int32_t)((fg & 0xFFFFu) << 8)) {
                        visible = false;
                        cast = false;
                    } else if (szp >= (int32_t)((fg >> 16) << 8)) {
                        cast = false;
                    }
                }
            }
            r.ox = sxp;
            r.oy = syp;
            r.oz = szp;
            r.dx = p.sun[0];
            r.dy = p.sun[1];
            r.dz = p.sun[2];
        }
        if (!__any_sync(kFull, cast)) break;
    }
    if (px >= (int32_t)c.w || py >= (int32_t)c.h) return;
    const uint32_t pix = (uint32_t)py * c.w + (uint32_t)px;
    const uint8_t face = tag & 0xFF;
    if (SHADOWS && c.shadow) __stcs(c.shadow + pix, (uint8_t)(visible ? 0 : 1));
    if (c.rgba)
        __stcs(c.rgba + pix, face < kFaceError ? shade(tag >> 8, face_cosine(face, p.sun_n), visible) : kSky);
}

// One warp renders one tile: lane l traces the tile's pixels l, l+32, ...
template <bool SHADOWS, bool PAIR, bool WIDE>
__device__ __forceinline__ void trace_tile(const RenderParams &p, const LevelDev *lvt,
                                           const BeamDir &sun, TileDev &t, uint32_t local_tile,
                                           int lane) {
    if (lane == 0) {
        t.x0 = (int32_t)(local_tile % t.cam.tiles_x) << p.tile_w_log2;
        t.y0 = (int32_t)(local_tile / t.cam.tiles_x) << p.tile_h_log2;
    }
    __syncwarp();
    for (int i = lane; i < 1 << (p.tile_w_log2 + p.tile_h_log2); i += 32)
        trace_pixels<SHADOWS, PAIR, WIDE>(p, lvt, t, i, sun);
}

// Copy camera i into this warp's shared slot.
__device__ __forceinline__ TileDev &stage_cam(TileDev *slot, const CamDev *cams, uint32_t i,
                                              int lane) {
    static_assert(sizeof(CamDev) % 4 == 0 && sizeof(CamDev) / 4 <= 32, "one word per lane");
    const uint32_t *src = reinterpret_cast<const uint32_t *>(cams + i);
    uint32_t *dst = reinterpret_cast<uint32_t *>(&slot->cam);
    __syncwarp();
    if (lane < (int)(sizeof(CamDev) / 4)) dst[lane] = src[lane];
    __syncwarp();
    return *slot;
}

// Persistent batched kernel: warps pop (camera, tile) items from one atomic
// counter until the batch is drained.  One launch renders every camera.
template <bool SHADOWS, bool PAIR>
__global__ void __launch_bounds__(kThreads, kTraceMinBlocks) k_trace_batched(const RenderParams p) {
    __shared__ uint32_t s_base[kMaxCams + 1];
    __shared__ TileDev s_tile[kThreads / 32];
    __shared__ LevelDev s_lv[kMaxLevels + 1];
    const uint32_t n = p.hdr->n_cams;
    const uint32_t total = p.hdr->total_tiles;
    __shared__ BeamDir s_sun;
    prefetch_world(p);
    if (SHADOWS && threadIdx.x == 32) s_sun = beam_dir(p.sun[0], p.sun[1], p.sun[2]);
    for (uint32_t i = threadIdx.x; i < n; i += blockDim.x) s_base[i] = p.cams[i].tile_base;
    fill_levels(s_lv, p.world);
    __syncthreads();
    const int lane = threadIdx.x & 31;
    for (;;) {
        uint32_t t = 0;
        if (lane == 0) t = atomicAdd(&p.hdr->counter, 1u);
        t = __shfl_sync(kFull, t, 0);
        if (t >= total) break;
        // last camera whose first tile is <= t
        uint32_t lo = 0, hi = n;
        while (hi - lo > 1) {
            const uint32_t mid = (lo + hi) >> 1;
            if (s_base[mid] <= t) lo = mid;
            else hi = mid;
        }
        TileDev &tile = stage_cam(&s_tile[threadIdx.x >> 5], p.cams, lo, lane);
        trace_tile<SHADOWS, PAIR, true>(p, s_lv, s_sun, tile, t - s_base[lo], lane);
    }
}

// Plain kernel: one camera, one warp per tile, grid covers the image once.
// The camera record is a kernel parameter, so a plain render needs no copy of
// it to the device; each warp stages it in shared memory like the batched
// kernel (reading the fields from parameter space instead changes the
// traversal's register allocation, measured 3-8 % slower on large images).
template <bool SHADOWS, bool PAIR>
__global__ void __launch_bounds__(kThreads, kTraceMinBlocks)
    k_trace_plain(const __grid_constant__ RenderParams p, const __grid_constant__ CamDev cam,
                  uint32_t n_tiles) {
    __shared__ LevelDev s_lv[kMaxLevels + 1];
    __shared__ TileDev s_tile[kThreads / 32];
    __shared__ BeamDir s_sun;
    prefetch_world(p);
    if (SHADOWS && threadIdx.x == 32) s_sun = beam_dir(p.sun[0], p.sun[1], p.sun[2]);
    fill_levels(s_lv, p.world);
    __syncthreads();
    const uint32_t t = blockIdx.x * (kThreads / 32) + (threadIdx.x >> 5);
    if (t >= n_tiles) return;
    const int lane = threadIdx.x & 31;
    TileDev &tile = stage_cam(&s_tile[threadIdx.x >> 5], &cam, 0, lane);
    trace_tile<SHADOWS, PAIR, false>(p, s_lv, s_sun, tile, t, lane);
}

template <bool SH, bool PA>
const void *batched_ptr() {
    return reinterpret_cast<const void *>(&k_trace_batched<SH, PA>);
}

}  // namespace

const void *trace_batched_fn(bool shadows, int kind, bool pair) {
    if (kind != kTraceBeams) return single_batched_fn(shadows, kind == kTraceStats, pair);
    if (shadows) return pair ? batched_ptr<true, true>() : batched_ptr<true, false>();
    return pair ? batched_ptr<false, true>() : batched_ptr<false, false>();
}

int trace_batched_occupancy(bool shadows, int kind, bool pair, int *blocks_per_sm) {
    cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(
        blocks_per_sm, trace_batched_fn(shadows, kind, pair), trace_threads(kind), 0);
    return e == cudaSuccess ? 0 : -1;
}

int launch_trace_batched(const RenderParams &p, bool shadows, int kind, int blocks, void *stream) {
    void *args[] = {const_cast<RenderParams *>(&p)};
    const cudaError_t e =
        cudaLaunchKernel(trace_batched_fn(shadows, kind, p.world.pair != 0), dim3(blocks),
                         dim3(trace_threads(kind)), args, 0, (cudaStream_t)stream);
    return e == cudaSuccess ? 0 : -1;
}

int launch_trace_plain(const RenderParams &p, bool shadows, int kind, const CamDev &cam,
                       uint32_t n_tiles, void *stream) {
    if (n_tiles == 0) return 0;
    if (kind != kTraceBeams)
        return launch_single_plain(p, shadows, kind == kTraceStats, cam, n_tiles, stream);
    cudaStream_t s = (cudaStream_t)stream;
    const uint32_t warps = kThreads / 32, blocks = (n_tiles + warps - 1) / warps;
    if (shadows && p.world.pair) k_trace_plain<true, true><<<blocks, kThreads, 0, s>>>(p, cam, n_tiles);
    else if (shadows) k_trace_plain<true, false><<<blocks, kThreads, 0, s>>>(p, cam, n_tiles);
    else if (p.world.pair) k_trace_plain<false, true><<<blocks, kThreads, 0, s>>>(p, cam, n_tiles);
    else k_trace_plain<false, false><<<blocks, kThreads, 0, s>>>(p, cam, n_tiles);
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

}  // namespace hf

// ------------------------------------------------------------------------
// Allocation-free render (hf_render_noalloc).  The paper has no counterpart:
// this exists for callers that must not allocate device memory once they are
// running (a render thread whose memory budget is fixed at start-up, or a
// loop where cudaMalloc/cudaFree would stall or implicitly synchronise the
// device).  hf_render may allocate its per-slot camera tables and CUDA graphs
// on first use or when a batch grows; this entry point never does.
//
// Its scratch -- the batch header with the tile counter, the camera table and
// the step-guard status word -- is one file-scope device array, present on
// every GPU that loads this library until the process exits.  Every call
// shares it and it keeps the last call's contents: each call rewrites the
// header (tile counter zero) and the camera table, and clears the status word,
// before its kernel runs.  Two calls whose work overlaps on the GPU race on
// this array; calls ordered on one stream do not.
namespace hf {
namespace {

constexpr size_t kNoallocCamOff = sizeof(BatchHeader);
constexpr size_t kNoallocStatusOff = kNoallocCamOff + (size_t)HF_NOALLOC_MAX_CAMERAS * sizeof(CamDev);
constexpr size_t kNoallocBytes = (kNoallocStatusOff + 64 + 255) & ~(size_t)255;
static_assert(kNoallocStatusOff % 8 == 0, "status words need 8-byte alignment");

static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoallocBytes];

constexpr int kMaxDevices = 64;
std::mutex g_noalloc_mu;
void *g_noalloc_ptr[kMaxDevices] = {};

// Device address of g_noalloc_scratch on the current device, looked up once
// per device.  In host code the array's name is only a host-side handle.
int noalloc_scratch(int device, void **out) {
    if (device < 0 || device >= kMaxDevices) return HF_E_CUDA;
    std::lock_guard<std::mutex> lock(g_noalloc_mu);
    if (!g_noalloc_ptr[device]) {
        void *ptr = nullptr;
        if (cudaGetSymbolAddress(&ptr, g_noalloc_scratch) != cudaSuccess || !ptr) {
            (void)cudaGetLastError();
            return HF_E_CUDA;
        }
        g_noalloc_ptr[device] = ptr;
    }
    *out = g_noalloc_ptr[device];
    return HF_OK;
}

int ilog2_pow2(uint32_t v) {
    if (v == 0 || (v & (v - 1))) return -1;
    int k = 0;
    while ((1u << k) < v) ++k;
    return k;
}

}  // namespace
}  // namespace hf

extern "C" int hf_render_noalloc(hf_ctx *ctx, const hf_camera *cams, uint32_t n,
                                 const hf_outputs *outs, const hf_render_opts *opts) {
    using namespace hf;
    if (!ctx) return HF_E_INVALID_ARG;
    if (n == 0) return HF_OK;
    if (!cams || !outs) return HF_E_INVALID_ARG;
    if (n > HF_NOALLOC_MAX_CAMERAS) return HF_E_INVALID_ARG;
    CtxView v;
    if (ctx_view(ctx, &v)) return HF_E_INVALID_ARG;
    hf_render_opts o;
    std::memset(&o, 0, sizeof(o));
    o.mip_start = HF_MIP_AUTO;
    if (opts) o = *opts;
    if (o.cuda_stream && o.cuda_stream != v.stream) return HF_E_INVALID_ARG;
    // a flag this entry point cannot honour (host outputs, statistics, plain
    // or graph launches, admission) is refused, not silently dropped
    if (o.flags & ~(HF_SHADOWS | HF_SYNC)) return HF_E_INVALID_ARG;
    const uint32_t tw = o.tile_w ? o.tile_w : 8, th = o.tile_h ? o.tile_h : 4;
    const int twl = ilog2_pow2(tw), thl = ilog2_pow2(th);
    if (twl < 0 || thl < 0 || tw * th < 32 || tw * th > 256 || tw > 256 || th > 256)
        return HF_E_INVALID_ARG;
    int32_t sun[3] = {o.sun[0], o.sun[1], o.sun[2]};
    if (sun[0] == 0 && sun[1] == 0 && sun[2] == 0) {
        sun[0] = 321060;
        sun[1] = -321060;
        sun[2] = 262144;
    }
    for (int i = 0; i < 3; ++i)
        if (sun[i] <= -(1 << 21) || sun[i] >= (1 << 21)) return HF_E_INVALID_ARG;

    // header + camera table, built on the stack (no allocation)
    alignas(16) unsigned char buf[kNoallocStatusOff];
    auto *hdr = reinterpret_cast<BatchHeader *>(buf);
    std::memset(hdr, 0, sizeof(*hdr));
    auto *cd = reinterpret_cast<CamDev *>(buf + kNoallocCamOff);
    for (uint32_t i = 0; i < n; ++i)
        if (hf_validate_camera((uint32_t)v.world.W, (uint32_t)v.world.H, &cams[i]) != HF_OK)
            return HF_E_INVALID_ARG;
    uint8_t wide[HF_NOALLOC_MAX_CAMERAS];
    const bool fit = beams_fit(v.world.W, v.world.H, cams, n, tw, kTraceShare, wide);
    uint64_t base = 0;
    uint32_t at = 0;
    for (const bool single : {true, false})  // wide views first, as in hf_render
        for (uint32_t i = 0; i < n; ++i) {
            const hf_camera &k = cams[i];
            if ((wide[i] != 0) != single) continue;
            CamDev &c = cd[at++];
            for (int a = 0; a < 3; ++a) {
                c.o[a] = (int32_t)k.origin[a];
                c.F[a] = k.fwd[a];
                c.R[a] = k.right[a];
                c.U[a] = k.up[a];
            }
            c.w = k.w;
            c.h = k.h;
            c.tiles_x = (k.w + tw - 1) / tw;
            c.single = single;
            c.tile_base = (uint32_t)base;
            base += (uint64_t)c.tiles_x * ((k.h + th - 1) / th);
            if (base >= 0xFFFFFFFFull) return HF_E_INVALID_ARG;
            c.hit_cell = outs[i].hit_cell;
            c.layer = outs[i].layer;
            c.face = outs[i].face;
            c.depth = outs[i].depth;
            c.rgba = outs[i].rgba;
            c.shadow = outs[i].shadow;
        }
    hdr->n_cams = n;
    hdr->total_tiles = (uint32_t)base;

    if (cudaSetDevice(v.device) != cudaSuccess) {
        (void)cudaGetLastError();
        return HF_E_CUDA;
    }
    void *scratch = nullptr;
    int rc = noalloc_scratch(v.device, &scratch);
    if (rc != HF_OK) return rc;
    unsigned char *sp = static_cast<unsigned char *>(scratch);
    cudaStream_t stream = (cudaStream_t)v.stream;
    const size_t bytes = kNoallocCamOff + (size_t)n * sizeof(CamDev);
    if (cudaMemcpyAsync(sp, buf, bytes, cudaMemcpyHostToDevice, stream) != cudaSuccess ||
        cudaMemsetAsync(sp + kNoallocStatusOff, 0, 64, stream) != cudaSuccess) {
        (void)cudaGetLastError();
        return HF_E_CUDA;
    }
    const bool shadows = (o.flags & HF_SHADOWS) != 0;
    const uint32_t mip = o.mip_start == HF_MIP_AUTO ? kDefaultMipStart : o.mip_start;
    const uint64_t guard = 4ull * ((uint64_t)v.world.W + (uint64_t)v.world.H) + 64;
    const uint32_t steps = o.max_steps ? o.max_steps : (uint32_t)guard;
    if (steps > 0x7FFFFFFFu) return HF_E_INVALID_ARG;
    RenderParams p;
    std::memset(&p, 0, sizeof(p));
    p.world = v.world;
    p.hdr = reinterpret_cast<BatchHeader *>(sp);
    p.cams = reinterpret_cast<const CamDev *>(sp + kNoallocCamOff);
    p.status = reinterpret_cast<uint32_t *>(sp + kNoallocStatusOff);
    p.stats = reinterpret_cast<unsigned long long *>(sp + kNoallocStatusOff + 8);
    p.tile_w_log2 = twl;
    p.tile_h_log2 = thl;
    p.mip_start = (int32_t)(mip > (uint32_t)v.world.L ? (uint32_t)v.world.L : mip);
    p.shadow_mip = (int32_t)((uint32_t)p.mip_start + kShadowMipExtra > (uint32_t)v.world.L
                                 ? (uint32_t)v.world.L
                                 : (uint32_t)p.mip_start + kShadowMipExtra);
    p.max_steps = (int32_t)steps;
    const double sn = sqrt((double)sun[0] * sun[0] + (double)sun[1] * sun[1] +
                           (double)sun[2] * sun[2]);
    for (int i = 0; i < 3; ++i) {
        p.sun[i] = sun[i];
        p.sun_n[i] = (float)(sun[i] / sn);
    }
    const int kind = o.max_steps || !fit ? kTraceGeneral : kTraceBeams;
    const int blocks = v.sm_count * v.occ[shadows ? 1 : 0][kind];
    if (launch_trace_batched(p, shadows, kind, blocks, stream)) return HF_E_CUDA;
    if (o.flags & HF_SYNC) {
        uint32_t status = 0;
        if (cudaMemcpyAsync(&status, p.status, sizeof(status), cudaMemcpyDeviceToHost, stream) !=
                cudaSuccess ||
            cudaStreamSynchronize(stream) != cudaSuccess) {
            (void)cudaGetLastError();
            return HF_E_CUDA;
        }
        if (status) return HF_E_STEP_LIMIT;
    }
    return HF_OK;
}
