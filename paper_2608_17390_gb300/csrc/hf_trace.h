// hf_trace.h -- what the kernels of beams (hf_trace.cu) and of single rays
// (hf_single.cu) have in common (device code).
#pragma once

#include "hf_cast.h"
#include "hf_internal.h"

namespace hf {
namespace {

__constant__ float c_albedo[8][3] = HF_ALBEDO_TABLE;
constexpr float kKa = kAmbient, kKd = kDiffuse;
constexpr uint32_t kSky = kSkyColour;

// int64 -> float through two 32-bit conversions (64-bit integer conversions
// run on the FP64 pipe, which is narrow on this GPU).  |v| < 2^52.
__device__ __forceinline__ float i64_to_f32(int64_t v) {
    return fmaf((float)(int32_t)(v >> 32), 4294967296.0f, (float)(uint32_t)v);
}

// floor(a / b) for |a| < 2^52, 0 < b < 2^21 and |a / b| < 2^30: a float
// estimate, a second estimate from the remainder, then one exact correction.
__device__ __forceinline__ int32_t floor_div_small(int64_t a, int32_t b, float rcp_b) {
    int32_t q = (int32_t)floorf(i64_to_f32(a) * rcp_b);        // within ~2^9 of the quotient
    const int32_t r1 = (int32_t)(a - (int64_t)q * b);          // |r1| < 2^31
    q += (int32_t)floorf((float)r1 * rcp_b);                   // within 1
    const int64_t r = a - (int64_t)q * b;
    if (r < 0) q -= 1;
    else if (r >= b) q += 1;
    return q;
}

// The colour of material m under the cosine ndl of the sun's angle.
__device__ __forceinline__ uint32_t shade(uint32_t m, float ndl, bool visible) {
    const float k = kKa + kKd * fmaxf(ndl, 0.0f) * (visible ? 1.0f : 0.0f);
    uint32_t out = 0xFF000000u;
#pragma unroll
    for (int ch = 0; ch < 3; ++ch) {
        const float v = fminf(fmaxf(c_albedo[m][ch] * k, 0.0f), 1.0f);
        out |= ((uint32_t)(255.0f * v + 0.5f)) << (8 * ch);
    }
    return out;
}

// Asks L2 for the world's coarse levels (all of a small world) as a launch
// starts, spread over all its threads.  A ray's fetches form one dependent
// chain, so a short render of a world that is not in L2 would otherwise wait
// on DRAM at every step of every ray.
__device__ __forceinline__ void prefetch_world(const RenderParams &p) {
    const uint32_t stride = gridDim.x * blockDim.x;
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < p.prefetch_lines; i += stride)
        asm volatile("prefetch.global.L2 [%0];" ::"l"(p.prefetch + (size_t)i * 32));
}

// stride of level 0 is its width in cells also for paired texels (whose rows
// then hold stride / 2 words)
__device__ __forceinline__ void fill_levels(LevelDev *s_lv, const WorldDev &w) {
    const int k = threadIdx.x;
    if (k <= w.L) s_lv[k] = LevelDev{w.base + w.off[k], (uint32_t)w.stride[k], (uint32_t)w.rows[k]};
}

}  // namespace
}  // namespace hf
