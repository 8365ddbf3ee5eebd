// hf_beam.h -- a warp's scan along a beam of its rays (device code; the parts
// are in hf_cast.h).
#pragma once

#include "hf_cast.h"

namespace hf {

constexpr uint32_t kFull = 0xFFFFFFFFu;

// (volatile: every lane must execute them together, so they stay where they are
// called, also where only some lanes go on to use the result)
__device__ __forceinline__ float warp_min(float v) {
    float r;
    asm volatile("redux.sync.min.f32 %0, %1, 0xffffffff;" : "=f"(r) : "f"(v));
    return r;
}
__device__ __forceinline__ float warp_max(float v) {
    float r;
    asm volatile("redux.sync.max.f32 %0, %1, 0xffffffff;" : "=f"(r) : "f"(v));
    return r;
}

// Rays that go the same way (key: the axis of the larger component and both
// signs) form a beam from mirrored cell (m.u0, m.v0) on.  Its 32 next stretches
// of columns are tested by the 32 lanes at once, each against the one to three
// nodes that the beam covers there; the runs of stretches that are not proven
// empty come out in order.
struct BeamScan {
    Beam m;
    int32_t key, limit;  // limit: the mirrored column past the grid
    float top;           // the world's highest top
    int base_level, top_level;
    // where the scan stands: columns before u are done; stretches j + i of
    // 2^level columns, bit i of `open` to come
    int32_t u, j;
    int level;
    uint32_t open;
    uint32_t high;       // the highest top in this lane's stretch
};

__device__ __forceinline__ void beam_scan(BeamScan &s, const WorldDev &w, const LevelDev *lvt,
                                          int mip) {
    s.limit = s.key & 2 ? 0 : (s.key & 4 ? w.W : w.H);
    s.top = (float)((cast_load(lvt[w.L].base) >> 16) & 0xFF);
    s.base_level = min(kBeamLevel, mip);
    s.top_level = min(kBeamTop, mip);
    s.u = s.m.u0;
    s.level = s.base_level;
    s.open = 0;
}

// The next run, columns [b0, b1), for the rays still alive (at least one); false
// when no more of the grid can hold a solid on their way.  All lanes call.
// SAMPLES: for the rounded samples on the rays (hf_march.h).
template <bool PAIR, bool SAMPLES = false>
__device__ __forceinline__ bool beam_next(BeamScan &s, const LevelDev *lvt, const BeamDir &d,
                                          const BeamRay &q, bool alive, int32_t &b0, int32_t &b1,
                                          uint32_t *peak = nullptr) {
    const int lane = threadIdx.x & 31;
    while (!s.open) {
        if (s.u >= s.limit) return false;
        {  // the beam of the rays that are left
            const float big = 3.0e38f;
            const float a = q.pv - d.rho * q.pu, b = q.z0 - d.sigma * q.pu;
            s.m.a0 = warp_min(alive ? a : big);
            s.m.a1 = warp_max(alive ? a : -big);
            s.m.r0 = warp_min(alive ? d.rho : big);
            s.m.r1 = warp_max(alive ? d.rho : -big);
            s.m.b0 = warp_min(alive ? b : big);
            s.m.b1 = warp_max(alive ? b : -big);
            s.m.s0 = warp_min(alive ? d.sigma : big);
            s.m.s1 = warp_max(alive ? d.sigma : -big);
        }
        s.u = beam_skip<SAMPLES>(s.m, s.u, s.limit, s.top);
        if (s.u >= s.limit) return false;
        const int least = beam_least(s.m, s.u, s.base_level, s.top_level);
        s.level = max(s.level, least);
        s.j = s.u >> s.level;
        const uint32_t open = __ballot_sync(
            kFull, beam_open<PAIR, SAMPLES>(lvt, s.m, s.level, s.j + lane, s.key, s.high));
        if (s.level > least && open) {
            s.u = max(s.u, (s.j + __ffs(open) - 1) * (1 << s.level));
            s.level = least;
        } else if (!open) {
            s.u = (s.j + 32) * (1 << s.level);
            s.level = min(s.level + 2, s.top_level);
        } else {
            s.open = SAMPLES ? beam_joined(open) : open;
        }
    }
    const int i = __ffs(s.open) - 1, run = beam_run(s.open, i);
    s.open &= i + run < 32 ? kFull << (i + run) : 0u;
    b0 = max(s.u, (s.j + i) * (1 << s.level));
    b1 = min((s.j + i + run) * (1 << s.level), s.limit);
    if (peak) *peak = __reduce_max_sync(kFull, lane >= i && lane < i + run ? s.high : 0u);
    if (!s.open) s.u = (s.j + 32) * (1 << s.level);
    return true;
}

}  // namespace hf
