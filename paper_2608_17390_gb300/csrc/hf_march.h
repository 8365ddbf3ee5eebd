// hf_march.h -- the samples of the fixed-step march, and which of them a beam's
// run of columns can hold.  Host code too, so that the march in beams can be
// compared with every sample on a CPU.
//
// A sample is off its ray.  Its position is rounded three times (the origin, the
// product t d, their sum), each by at most 2^-11 on x and y (up to 16384 cells)
// and 2^-13 on the height (up to 4096): by less than 2^-9 and 2^-11 in all.  Beams
// tell heights and rows by the column, so an error along the columns counts with
// the ray's slope: on a ray that falls 1000 units a column, 2^-9 columns are two
// units of height.  What covers it (kSampleAlong in hf_cast.h): slopes times 2^-8
// in the height slack, as a sample may also lie before the start; the scan begins
// one column before the start's; a run's samples have 0.02 columns more at either
// end, and one that lies in the column after the run is left to the next.
#pragma once

#include "hf_cast.h"

namespace hf {

// Rounded once each, never fused.
HF_HD float rn_mul(float a, float b) {
#ifdef __CUDA_ARCH__
    return __fmul_rn(a, b);
#else
    return a * b;
#endif
}
HF_HD float rn_add(float a, float b) {
#ifdef __CUDA_ARCH__
    return __fadd_rn(a, b);
#else
    return a + b;
#endif
}

// A pixel ray in float; sample i lies at t = i dt, i = 1 .. steps.
struct MarchRay {
    float ox, oy, oz, dx, dy, dz, dt;
};

struct MarchSpot {
    int32_t cx, cy;
    float z;
};
HF_HD MarchSpot march_spot(const MarchRay &m, float t) {
    MarchSpot s;
    s.cx = (int32_t)floorf(rn_add(m.ox, rn_mul(t, m.dx)));
    s.cy = (int32_t)floorf(rn_add(m.oy, rn_mul(t, m.dy)));
    s.z = rn_add(m.oz, rn_mul(t, m.dz));
    return s;
}

// Whether height z is solid in the cell of a node-form word.  (Both intervals are
// tested: with the second only where the first fails, 390 renders that take every
// sample took 2.5 % longer on the average.)
HF_HD bool march_solid(uint32_t c, float z, bool &floor_) {
    const uint32_t h0 = c & 0xFF, h1 = (c >> 8) & 0xFF, h2 = (c >> 16) & 0xFF;
    floor_ = z <= (float)h0;
    const bool upper = h2 > h0 && z >= (float)h1 && z <= (float)h2;
    return floor_ || upper;
}

// The mirrored column of a cell for a beam's key.
HF_HD int32_t march_column(const MarchSpot &s, int32_t key) {
    const int32_t c = key & 4 ? s.cx : s.cy;
    return key & 2 ? ~c : c;
}

// Samples per column and per unit of height.
struct MarchRate {
    float u, z;
};
HF_HD MarchRate march_rate(const MarchRay &m, const BeamDir &d) {
#ifdef __CUDA_ARCH__
    return MarchRate{__fdividef(65536.0f, (float)d.du * m.dt),
                     __fdividef(1.0f, fabsf(m.dz) * m.dt)};
#else
    return MarchRate{65536.0f / ((float)d.du * m.dt), 1.0f / (fabsf(m.dz) * m.dt)};
#endif
}

// The samples first .. last that can be solid in a run's columns, x0 up to x1 past
// the beam's cell, whose highest top is peak: a little more either side than
// rounding can move them.  Those before `done` lie before x1 in any case.  past:
// the run lies beyond the last sample.
struct MarchRun {
    int32_t first, last, done;
    bool past;
};
HF_HD MarchRun march_run(const MarchRay &m, const MarchRate &r, float pu, float x0, float x1,
                         float peak, float steps) {
    MarchRun w;
    float lo = (x0 - 0.02f - pu) * r.u;
    float hi = (x1 + 0.02f - pu) * r.u;
    w.past = lo * 0.999998f - 0.02f > steps;
    const float rise = peak + 0.02f - m.oz;
    if (m.dz < 0.0f) lo = fmaxf(lo, -rise * r.z);
    else hi = fminf(hi, rise * r.z);
    lo = fminf(fmaxf(lo * (lo > 0.0f ? 0.999998f : 1.0f) - 0.02f, 0.0f), steps + 1.0f);
    hi = fminf(fmaxf(hi * 1.000002f + 0.02f, 0.0f), steps);
    const float done = (x1 - 0.02f - pu) * r.u * 0.999998f - 0.02f;
    w.first = (int32_t)lo;
    w.last = (int32_t)hi;
    w.done = (int32_t)fminf(fmaxf(done, 0.0f), steps + 1.0f);
    return w;
}

}  // namespace hf
