// hf_march.cu -- the paper's fixed-step height-field ray march (its Section
// 3.1), as a comparison kernel for the exact cast.
//
// Per pixel ray p(t) = o + t d in world units (o = origin / 2^16, d = integer
// direction / 2^16, the same parameter t as the exact cast): the segment is
// clipped at the far distance and, for a descending ray, at z = 0; `steps`
// samples are spaced uniformly over it; the first sample whose point is solid
// (z <= low, or mid <= z <= high, of the cell containing it) stops the search
// and `bisections` halvings keep the solid end.  A ray with no solid sample
// misses.  All arithmetic is float32, round to nearest, with no fused
// multiply-add, in a fixed order, so results are reproducible bit for bit.
// The method can step over features thinner than its sample spacing (the
// trade-off the paper states); the exact cast cannot.
//
// Samples that cannot be solid are not taken: the 32 rays of a warp are bounded
// by beams as in the exact cast (hf_beam.h), and only samples whose column lies
// in a stretch that the beam does not prove empty, at a height that its cells
// reach, are looked up (hf_march.h: the bounds of their rounding).
// Bound by instruction issue: 12 views of 1280 x 800 over 2048 x 16384 cells, 128
// samples a ray, 1.229 -> 0.608 ms.
#include <cuda_runtime.h>

#include "hf_beam.h"
#include "hf_internal.h"
#include "hf_march.h"

namespace hf {
namespace {

constexpr int kMarchThreads = 128;
// Nine blocks leave each thread 56 registers.  12 views of 1280 x 800 with 128
// samples a ray: seven blocks 638 us, nine 622, eleven (46 registers) 692.
constexpr int kMarchMinBlocks = 9;
// The kernel that takes every sample (hf_rules.h says when) needs 40 registers, so
// that six blocks fit an SM (asked for, they cost it 0.6 %); in blocks of 128 threads
// it is 3 % slower.
constexpr int kMarchAllBlocks = 6, kMarchAllThreads = 256;

struct MarchPoint {
    bool solid;
    MarchSpot at;
    uint8_t layer;
};

__device__ __forceinline__ MarchPoint march_at(const WorldDev &w, const MarchRay &m, float t) {
    MarchPoint r;
    r.at = march_spot(m, t);
    r.solid = false;
    r.layer = 0;
    if ((uint32_t)r.at.cx < (uint32_t)w.W && (uint32_t)r.at.cy < (uint32_t)w.H) {
        bool floor_;
        r.solid = march_solid(level0_node(w, r.at.cx, r.at.cy), r.at.z, floor_);
        r.layer = floor_ ? 0 : 1;
    }
    return r;
}

// The first solid sample of each active lane's ray among i .. last, or 0.
// Every lane of the warp calls.
__device__ __forceinline__ int32_t march_samples(const WorldDev &w, const MarchRay &m, bool active,
                                                 int32_t i, int32_t last) {
    int32_t found = 0;
    bool go = active && i <= last;
    while (__any_sync(kFull, go)) {
        if (go) {
            if (march_at(w, m, __fmul_rn((float)i, m.dt)).solid) found = i;
            go = !found && i < last;
            ++i;
        }
    }
    return found;
}

// The first solid sample of each lane's ray, or 0; every lane of the warp calls.
__device__ __forceinline__ int32_t march_beams(const RenderParams &p, const MarchParams &mp,
                                               const LevelDev *lvt, const Ray &r, const MarchRay &m,
                                               bool inside, bool single) {
    int32_t found = 0;
    const int lane = threadIdx.x & 31;
    const BeamDir d = beam_dir(r.dx, r.dy, r.dz);
    BeamRay q = beam_ray(d, r);
    const MarchRate rate = march_rate(m, d);
    const float steps = (float)mp.steps;
    // every sample of a wide view's rays, and of a ray that is vertical or whose
    // spacing is no ordinary number
    const bool plain = single || d.du == 0 || !(m.dt > 1e-9f && m.dt < 1e9f);
    uint32_t todo = __ballot_sync(kFull, inside && !plain);
    while (todo) {
        const int lead = __ffs(todo) - 1;
        BeamScan s;
        s.key = __shfl_sync(kFull, d.key, lead);
        s.m.u0 = __shfl_sync(kFull, q.fu, lead);  // (one start for all rays)
        s.m.v0 = __shfl_sync(kFull, q.fv, lead);
        bool alive = (todo >> lane & 1) && d.key == s.key;
        todo &= ~__ballot_sync(kFull, alive);
        beam_scan(s, p.world, lvt, p.world.L);
        s.u = s.m.u0 - 1;  // (rounding may put samples there)
        beam_place(q, s.m);
        int32_t next = 1, b0, b1;
        uint32_t peak;
        while (beam_next<false, true>(s, lvt, d, q, alive, b0, b1, &peak)) {
            const MarchRun run = march_run(m, rate, q.pu, (float)(b0 - s.m.u0),
                                           (float)(b1 - s.m.u0), (float)peak, steps);
            alive = alive && !run.past;
            const int32_t i = march_samples(p.world, m, alive, max(next, run.first), run.last);
            // one in the column beyond, which may be higher, is met again there
            if (i && march_column(march_spot(m, rn_mul((float)i, m.dt)), s.key) < b1) found = i;
            next = max(next, run.done);
            alive = alive && !found;
            if (!__any_sync(kFull, alive)) break;
        }
    }
    if (__any_sync(kFull, inside && plain))
        found = max(found, march_samples(p.world, m, inside && plain, 1, mp.steps));
    return found;
}

// The ray of a pixel, its samples and its length.
__device__ __forceinline__ MarchRay march_ray(const MarchParams &mp, const Ray &r, float &len) {
    const float inv_s = 1.0f / 65536.0f;
    MarchRay m;
    m.ox = __fmul_rn(__int2float_rn(r.ox), inv_s);
    m.oy = __fmul_rn(__int2float_rn(r.oy), inv_s);
    m.oz = __fmul_rn(__int2float_rn(r.oz), inv_s);
    m.dx = __fmul_rn(__int2float_rn(r.dx), inv_s);
    m.dy = __fmul_rn(__int2float_rn(r.dy), inv_s);
    m.dz = __fmul_rn(__int2float_rn(r.dz), inv_s);
    float sq = __fmul_rn(m.dx, m.dx);
    sq = __fadd_rn(sq, __fmul_rn(m.dy, m.dy));
    sq = __fadd_rn(sq, __fmul_rn(m.dz, m.dz));
    len = __fsqrt_rn(sq);
    float t_end = __fdiv_rn(mp.far_dist, len);
    if (m.dz < 0.0f) {
        const float tz = __fdiv_rn(-m.oz, m.dz);
        if (tz < t_end) t_end = tz;
    }
    m.dt = __fdiv_rn(t_end, (float)(mp.steps + 1));
    return m;
}

// A pixel's outputs: found says whether the sample at tb is its first solid one;
// ta: the sample before.
__device__ __forceinline__ void march_store(const RenderParams &p, const MarchParams &mp,
                                            const CamDev &c, int32_t px, int32_t py,
                                            const MarchRay &m, float len, bool found, float ta,
                                            float tb) {
    uint32_t cell = 0xFFFFFFFFu;
    uint8_t layer = 255;
    float depth = __int_as_float(0x7f800000);
    if (found) {
        for (int k = 0; k < mp.bisections; ++k) {
            const float tm = __fmul_rn(__fadd_rn(ta, tb), 0.5f);
            if (march_at(p.world, m, tm).solid) tb = tm;
            else ta = tm;
        }
        const MarchPoint hit = march_at(p.world, m, tb);
        cell = (uint32_t)hit.at.cy * (uint32_t)p.world.W + (uint32_t)hit.at.cx;
        layer = hit.layer;
        depth = __fmul_rn(tb, len);
    }
    const uint32_t pix = (uint32_t)py * c.w + (uint32_t)px;
    if (c.hit_cell) __stcs(c.hit_cell + pix, cell);
    if (c.layer) __stcs(c.layer + pix, layer);
    if (c.depth) __stcs(c.depth + pix, depth);
}

// One pixel per lane; every lane of the warp calls.
__device__ __forceinline__ void march_pixels(const RenderParams &p, const MarchParams &mp,
                                             const LevelDev *lvt, const CamDev &c, int32_t px,
                                             int32_t py) {
    const bool inside = px < (int32_t)c.w && py < (int32_t)c.h;
    const Ray r = primary_ray(c, px, py);
    float len;
    const MarchRay m = march_ray(mp, r, len);
    const int32_t i = march_beams(p, mp, lvt, r, m, inside, c.single != 0);
    if (inside)
        march_store(p, mp, c, px, py, m, len, i != 0, __fmul_rn((float)(i - 1), m.dt),
                    __fmul_rn((float)i, m.dt));
}

// One pixel of a lane that takes every sample.
__device__ __forceinline__ void march_pixel(const RenderParams &p, const MarchParams &mp,
                                            const CamDev &c, int32_t px, int32_t py) {
    if (px >= (int32_t)c.w || py >= (int32_t)c.h) return;
    float len;
    const MarchRay m = march_ray(mp, primary_ray(c, px, py), len);
    bool found = false;
    float ta = 0.0f, tb = 0.0f;
    for (int i = 1; i <= mp.steps; ++i) {
        const float t = __fmul_rn((float)i, m.dt);
        if (march_at(p.world, m, t).solid) {
            found = true;
            tb = t;
            ta = __fmul_rn((float)(i - 1), m.dt);
            break;
        }
    }
    march_store(p, mp, c, px, py, m, len, found, ta, tb);
}

__device__ __forceinline__ const CamDev &stage(CamDev *slot, const CamDev *cams, uint32_t i,
                                               int lane) {
    const uint32_t *src = reinterpret_cast<const uint32_t *>(cams + i);
    uint32_t *dst = reinterpret_cast<uint32_t *>(slot);
    __syncwarp();
    if (lane < (int)(sizeof(CamDev) / 4)) dst[lane] = src[lane];
    __syncwarp();
    return *slot;
}

// Persistent: warps pop (camera, tile) items from the batch's atomic counter.
template <bool BEAMS>
__global__ void __launch_bounds__(BEAMS ? kMarchThreads : kMarchAllThreads,
                                  BEAMS ? kMarchMinBlocks : 1)
    k_march_batched(const RenderParams p, const MarchParams m) {
    __shared__ LevelDev s_lv[kMaxLevels + 1];
    __shared__ uint32_t s_base[kMaxCams + 1];
    __shared__ CamDev s_cam[(BEAMS ? kMarchThreads : kMarchAllThreads) / 32];
    const uint32_t n = p.hdr->n_cams;
    const uint32_t total = p.hdr->total_tiles;
    for (uint32_t i = threadIdx.x; i < n; i += blockDim.x) s_base[i] = p.cams[i].tile_base;
    if (BEAMS && threadIdx.x <= (unsigned)p.world.L) {
        const int l = threadIdx.x;
        s_lv[l] = LevelDev{p.world.base + p.world.off[l], p.world.stride[l], p.world.rows[l]};
    }
    __syncthreads();
    const int lane = threadIdx.x & 31;
    for (;;) {
        uint32_t t = 0;
        if (lane == 0) t = atomicAdd(&p.hdr->counter, 1u);
        t = __shfl_sync(0xFFFFFFFFu, t, 0);
        if (t >= total) break;
        uint32_t lo = 0, hi = n;
        while (hi - lo > 1) {
            const uint32_t mid = (lo + hi) >> 1;
            if (s_base[mid] <= t) lo = mid;
            else hi = mid;
        }
        const CamDev &c = stage(&s_cam[threadIdx.x >> 5], p.cams, lo, lane);
        const uint32_t local = t - s_base[lo];
        const uint32_t tx = local % c.tiles_x, ty = local / c.tiles_x;
        const int32_t x0 = (int32_t)tx << p.tile_w_log2, y0 = (int32_t)ty << p.tile_h_log2;
        const int32_t npix = 1 << (p.tile_w_log2 + p.tile_h_log2);
        for (int i = lane; i < npix; i += 32) {
            const int32_t px = x0 + (i & ((1 << p.tile_w_log2) - 1));
            const int32_t py = y0 + (i >> p.tile_w_log2);
            if (BEAMS) march_pixels(p, m, s_lv, c, px, py);
            else march_pixel(p, m, c, px, py);
        }
    }
}

}  // namespace

// blocks: as many as are resident of the kernel with beams (march_occupancy).
int launch_march_batched(const RenderParams &p, const MarchParams &m, bool beams, int blocks,
                         void *stream) {
    cudaStream_t s = (cudaStream_t)stream;
    if (beams) {
        k_march_batched<true><<<blocks, kMarchThreads, 0, s>>>(p, m);
    } else {
        const int all = (blocks * kMarchAllBlocks + kMarchMinBlocks - 1) / kMarchMinBlocks;
        k_march_batched<false><<<all, kMarchAllThreads, 0, s>>>(p, m);
    }
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

int march_occupancy(int *blocks_per_sm) {
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(
               blocks_per_sm, reinterpret_cast<const void *>(&k_march_batched<true>), kMarchThreads, 0) ==
                   cudaSuccess
               ? 0
               : -1;
}

}  // namespace hf
