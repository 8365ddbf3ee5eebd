// hf_scatter.cu -- the paper's Scattered method (its Section 3: the original
// engine's object-order painter recast as a parallel atomic scatter), as a
// comparison renderer for the exact cast.
//
// Per camera, a grid of nu x nv samples covers a camera-aligned ground
// footprint (longitudinal coordinate s along the camera's horizontal forward,
// quadratically warped so samples crowd near the camera; lateral coordinate u
// along its right vector, |u| <= u_min + k_lat |s|: a trapezoid).  Each sample walks the
// column of the cell under it -- nz points from the floor top down to 0, and
// for a slab nz points from its top down to its underside -- projects each
// point with the integer camera basis (d = F + aR + bU), and keeps, per pixel,
// the minimum of (24-bit quantised Euclidean depth << 8 | material | layer << 3)
// with a 32-bit atomicMin (the paper's packing).  A resolve pass then turns
// each pixel's word into a depth, the cell under the reconstructed point, the
// layer and a colour.  Sampling leaves gaps where the footprint is sparse: the
// trade-off the paper measures with its coherence metric.
//
// All arithmetic is float32, round to nearest, no fused multiply-add, in a
// fixed order, so the result is reproducible bit for bit (the packed screen
// does not depend on the order of the atomics: min is order-free).
#include <cuda_runtime.h>

#include "hf_internal.h"

namespace hf {
namespace {

constexpr uint32_t kEmpty = 0xFFFFFFFFu;
constexpr float kQMax = 16777215.0f;  // 2^24 - 1
constexpr int kScatterThreads = 256;

// float32 camera constants, computed in the definition's order
struct ScatterCam {
    float ox, oy, oz;
    float Fx, Fy, Fz, Rx, Ry, Rz, Ux, Uy, Uz;
    float cF, cR, cU;
    float rhx, rhy, fhx, fhy;
};

__device__ __forceinline__ float inv_sq(float x, float y, float z) {
    return __fdiv_rn(1.0f, __fadd_rn(__fadd_rn(__fmul_rn(x, x), __fmul_rn(y, y)), __fmul_rn(z, z)));
}

__device__ __forceinline__ ScatterCam scatter_cam(const CamDev &c) {
    ScatterCam k;
    const float inv_s = 1.0f / 65536.0f;
    k.ox = __fmul_rn(__int2float_rn(c.o[0]), inv_s);
    k.oy = __fmul_rn(__int2float_rn(c.o[1]), inv_s);
    k.oz = __fmul_rn(__int2float_rn(c.o[2]), inv_s);
    k.Fx = (float)c.F[0];  // |components| < 2^21: exact
    k.Fy = (float)c.F[1];
    k.Fz = (float)c.F[2];
    k.Rx = (float)c.R[0];
    k.Ry = (float)c.R[1];
    k.Rz = (float)c.R[2];
    k.Ux = (float)c.U[0];
    k.Uy = (float)c.U[1];
    k.Uz = (float)c.U[2];
    k.cF = inv_sq(k.Fx, k.Fy, k.Fz);
    k.cR = inv_sq(k.Rx, k.Ry, k.Rz);
    k.cU = inv_sq(k.Ux, k.Uy, k.Uz);
    const float lr = __fsqrt_rn(__fadd_rn(__fmul_rn(k.Rx, k.Rx), __fmul_rn(k.Ry, k.Ry)));
    k.rhx = __fdiv_rn(k.Rx, lr);
    k.rhy = __fdiv_rn(k.Ry, lr);
    k.fhx = -k.rhy;
    k.fhy = k.rhx;
    return k;
}

__device__ __forceinline__ float dot3(float ax, float ay, float az, float bx, float by, float bz) {
    return __fadd_rn(__fadd_rn(__fmul_rn(ax, bx), __fmul_rn(ay, by)), __fmul_rn(az, bz));
}

// The parts of a point's view-space products that do not depend on its
// height: for v = (vx, vy, vz), dot3(v, a) = (vx ax + vy ay) + vz az, and the
// bracket is the same for every point of one column.
struct ColumnPartials {
    float vx, vy, pf, pr, pu, pd;
};

__device__ __forceinline__ ColumnPartials column_partials(const ScatterCam &k, float x, float y) {
    ColumnPartials c;
    c.vx = __fsub_rn(x, k.ox);
    c.vy = __fsub_rn(y, k.oy);
    c.pf = __fadd_rn(__fmul_rn(c.vx, k.Fx), __fmul_rn(c.vy, k.Fy));
    c.pr = __fadd_rn(__fmul_rn(c.vx, k.Rx), __fmul_rn(c.vy, k.Ry));
    c.pu = __fadd_rn(__fmul_rn(c.vx, k.Ux), __fmul_rn(c.vy, k.Uy));
    c.pd = __fadd_rn(__fmul_rn(c.vx, c.vx), __fmul_rn(c.vy, c.vy));
    return c;
}

// 1 / v with a relative error below 2^-22.
__device__ __forceinline__ float scatter_rcp(float v) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(v));
    return r;
}

// floor((n / den + size) / 2) with n / den rounded, or that with the quotient
// subtracted (flip): the pixel index of one axis, true if it is in [0, size).
// The quotient by way of r = 1 / den is off by less than 2^-22.4 of itself, and
// so half its sum with size by less than e; the index is certain unless the sum
// lies that near to a whole number: only then (one point in some hundreds) is
// the rounded division made.  The floor is taken by adding 1.5 2^23, whose
// neighbours are whole numbers, to the sum less 1/2.
__device__ __forceinline__ bool pixel_index(float n, float den, float r, float size, bool flip,
                                            uint32_t &index) {
    constexpr float kWhole = 12582912.0f;  // 1.5 2^23
    const float q = __fmul_rn(n, r);
    const float v = fmaf(flip ? -0.5f : 0.5f, q, 0.5f * size - 0.5f);
    const float b = __fadd_rn(v, kWhole);
    float f = __fsub_rn(b, kWhole);
    const float e = fmaf(fabsf(q), 1.0f / 4194304.0f, size * (1.0f / 4194304.0f));
    index = __float_as_uint(b) - __float_as_uint(kWhole);
    if (!(fabsf(v - f) < 0.5f - e)) {
        const float a = __fdiv_rn(n, den);
        f = floorf(__fmul_rn(flip ? __fsub_rn(size, a) : __fadd_rn(a, size), 0.5f));
        index = (uint32_t)f;
    }
    return f >= 0.0f && f < size;
}

// Packed depth word of a point without its type, or false when the point is
// behind the camera or outside the image.  The same operations, in the same
// order, as dot3 over the full vectors.
__device__ __forceinline__ bool project(const ScatterCam &k, float wf, float hf, uint32_t w,
                                        float qscale, const ColumnPartials &cp, float z,
                                        uint32_t &pix, uint32_t &q) {
    const float vz = __fsub_rn(z, k.oz);
    const float vf = __fadd_rn(cp.pf, __fmul_rn(vz, k.Fz));
    const float vr = __fadd_rn(cp.pr, __fmul_rn(vz, k.Rz));
    const float vu = __fadd_rn(cp.pu, __fmul_rn(vz, k.Uz));
    const float den = __fmul_rn(vf, k.cF), r = scatter_rcp(den);
    uint32_t px, py;
    const bool in_x = pixel_index(__fmul_rn(vr, k.cR), den, r, wf, false, px);
    const bool in_y = pixel_index(__fmul_rn(vu, k.cU), den, r, hf, true, py);
    if (!(vf > 0.0f && in_x && in_y)) return false;
    const float d = __fsqrt_rn(__fadd_rn(cp.pd, __fmul_rn(vz, vz)));
    q = __float2uint_rz(fminf(__fmul_rn(d, qscale), kQMax));
    pix = py * w + px;
    return true;
}

// Narrows [za, zb] to where the linear function that is g0 at z = 0 and g1 at
// z = 256 may be at least 0; e: a bound of what g0 and g1 are off.
__device__ __forceinline__ void clip_heights(float g0, float g1, float e, float &za, float &zb) {
    g0 += e;
    g1 += e;
    if (g0 < 0.0f && g1 < 0.0f) zb = -1.0f;  // nowhere
    const float z = 256.0f * __fdividef(g0, g0 - g1);
    if (g0 < 0.0f && g1 >= 0.0f) za = fmaxf(za, z);
    if (g1 < 0.0f && g0 >= 0.0f) zb = fminf(zb, z);
}

// The heights [za, zb] of a column that can lie inside the image (zb < za: none
// does).  A point does when vf > 0 and |n_r| <= w den, |n_u| <= h den (to less
// than a pixel), all linear in its height.  e is some 50 times what rounding
// can move these by, so the computed range holds the true one.
__device__ __forceinline__ void visible_heights(const ScatterCam &k, const ColumnPartials &cp,
                                                float wf, float hf, float &za, float &zb) {
    const float v0 = -k.oz, v1 = 256.0f - k.oz;
    const float f0 = fmaf(v0, k.Fz, cp.pf), f1 = fmaf(v1, k.Fz, cp.pf);
    const float d0 = f0 * k.cF, d1 = f1 * k.cF;
    const float r0 = fmaf(v0, k.Rz, cp.pr) * k.cR, r1 = fmaf(v1, k.Rz, cp.pr) * k.cR;
    const float u0 = fmaf(v0, k.Uz, cp.pu) * k.cU, u1 = fmaf(v1, k.Uz, cp.pu) * k.cU;
    // magnitudes of the terms, not of their sums, bound the rounding
    const float far = fabsf(k.oz) + 256.0f;
    const float mf = (fabsf(cp.vx * k.Fx) + fabsf(cp.vy * k.Fy) + far * fabsf(k.Fz)) * k.cF;
    const float mr = (fabsf(cp.vx * k.Rx) + fabsf(cp.vy * k.Ry) + far * fabsf(k.Rz)) * k.cR;
    const float mu = (fabsf(cp.vx * k.Ux) + fabsf(cp.vy * k.Uy) + far * fabsf(k.Uz)) * k.cU;
    const float w2 = wf + 2.0f, h2 = hf + 2.0f;
    const float ew = 1e-5f * (mr + w2 * mf), eh = 1e-5f * (mu + h2 * mf);
    za = 0.0f;
    zb = 256.0f;
    clip_heights(d0, d1, 1e-5f * mf, za, zb);
    clip_heights(w2 * d0 + r0, w2 * d1 + r1, ew, za, zb);
    clip_heights(w2 * d0 - r0, w2 * d1 - r1, ew, za, zb);
    clip_heights(h2 * d0 + u0, h2 * d1 + u1, eh, za, zb);
    clip_heights(h2 * d0 - u0, h2 * d1 - u1, eh, za, zb);
}

// The points m of an interval from `top` down to `bottom`, nz of them, whose
// heights can lie in [za, zb]: [m0, m1), one more at either end.
__device__ __forceinline__ void visible_points(float top, float bottom, float za, float zb,
                                               uint32_t nz, uint32_t &m0, uint32_t &m1) {
    m0 = 0;
    m1 = 0;
    if (!(zb >= za) || za > top + 0.01f || zb < bottom - 0.01f) return;
    if (top == bottom) {  // one point, nz times
        m1 = 1;
        return;
    }
    const float per = __fdividef((float)(nz - 1), top - bottom);
    const float a = floorf((top - zb) * per) - 1.0f, b = ceilf((top - za) * per) + 2.0f;
    m0 = a > 0.0f ? (uint32_t)a : 0u;
    m1 = b < (float)nz ? (uint32_t)fmaxf(b, 0.0f) : nz;
}

constexpr int kScatterMaxPoints = 4096;  // largest nz

__global__ void k_scatter_clear(const RenderParams p) {
    const CamDev &c = p.cams[blockIdx.y];
    const uint32_t n = c.w * c.h;
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
        c.hit_cell[i] = kEmpty;
}

// One thread per footprint sample: the column's heights that the image can
// hold, then the points there.  About half of the footprint's points miss the
// image, most of them whole columns.
//
// Bound by instruction issue: 280 warp instructions to place a column and clip
// it, 72 a point.  12 views of 1280 x 800, 1024 x 1024 samples of 16 points:
// about 480 us; 693 us with every point projected, by two rounded divisions.  (The first
// thread of a warp of its own makes the camera's terms: with the first thread of
// the table's, renders took 1.6 % longer on the average.)
//
// FEW: a launch that leaves most of the GPU idle is bound by the latency of a
// thread's points instead.  Floor and slab take their points in one loop then, so
// that one's work goes on while the other's waits: 64 x 64 samples of 1000 points
// 634 -> 530 us, 256 x 256 of 32 over paired texels 41 -> 37.  Where warps abound
// the loop of both costs 3 to 5 % (a slab's lanes hold up the others' floors).
template <bool FEW>
__global__ void __launch_bounds__(kScatterThreads) k_scatter(const RenderParams p,
                                                             const ScatterParams s) {
    __shared__ float s_tm[kScatterMaxPoints];  // column fractions m / (nz - 1)
    __shared__ ScatterCam s_cam;
    const float zden = (float)(s.nz - 1);
    const uint32_t cam = blockIdx.y;
    const CamDev &c = p.cams[cam];
    for (uint32_t m = threadIdx.x; m < s.nz; m += blockDim.x)
        s_tm[m] = __fdiv_rn((float)m, zden);
    if (threadIdx.x == 32) s_cam = scatter_cam(c);
    __syncthreads();
    const float4 fp = reinterpret_cast<const float4 *>(p.cams + p.hdr->n_cams)[cam];
    const uint32_t idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= s.nu * s.nv) return;
    const uint32_t i = idx % s.nu, j = idx / s.nu;
    const ScatterCam k = s_cam;
    // footprint sample (i, j)
    const float t = __fdiv_rn(__fadd_rn((float)j, 0.5f), (float)s.nv);
    const float sl = __fadd_rn(fp.x, __fmul_rn(__fsub_rn(fp.y, fp.x), __fmul_rn(t, t)));
    const float half = __fadd_rn(fp.w, __fmul_rn(fabsf(sl), fp.z));
    const float ui = __fsub_rn(__fmul_rn(__fdiv_rn(__fadd_rn((float)i, 0.5f), (float)s.nu), 2.0f), 1.0f);
    const float u = __fmul_rn(half, ui);
    const float x = __fadd_rn(__fadd_rn(k.ox, __fmul_rn(sl, k.fhx)), __fmul_rn(u, k.rhx));
    const float y = __fadd_rn(__fadd_rn(k.oy, __fmul_rn(sl, k.fhy)), __fmul_rn(u, k.rhy));
    const float fx = floorf(x), fy = floorf(y);
    if (!(fx >= 0.0f && fx < (float)p.world.W && fy >= 0.0f && fy < (float)p.world.H)) return;
    const float wf = (float)c.w, hf = (float)c.h;
    const uint32_t w = c.w;
    const ColumnPartials cp = column_partials(k, x, y);
    float za, zb;
    visible_heights(k, cp, wf, hf, za, zb);
    if (!(zb >= za)) return;
    const uint32_t node = level0_node(p.world, (int32_t)fx, (int32_t)fy);
    const uint32_t b0 = node & 0xFF, b1 = (node >> 8) & 0xFF, b2 = (node >> 16) & 0xFF;
    const uint32_t mat = (node >> 24) & 7;
    const bool slab = b2 > b0;  // node form: a slab exactly when its top is above the floor
    const float h0 = (float)b0, h1 = (float)b1, h2 = (float)b2;
    const float qscale = s.qscale;
    uint32_t *buf = c.hit_cell;
    uint32_t m0, m1, s0 = 0, s1 = 0, pix, q;
    visible_points(h0, 0.0f, za, zb, s.nz, m0, m1);
    auto floor_point = [&](uint32_t m) {
        if (project(k, wf, hf, w, qscale, cp, __fsub_rn(h0, __fmul_rn(h0, s_tm[m])), pix, q))
            atomicMin(buf + pix, (q << 8) | mat);
    };
    auto slab_point = [&](uint32_t m) {
        if (project(k, wf, hf, w, qscale, cp,
                    __fadd_rn(h2, __fmul_rn(__fsub_rn(h1, h2), s_tm[m])), pix, q))
            atomicMin(buf + pix, (q << 8) | mat | 8u);
    };
    if (FEW) {
        if (slab) visible_points(h2, h1, za, zb, s.nz, s0, s1);
        for (uint32_t m = m1 ? (s1 ? min(m0, s0) : m0) : s0; m < max(m1, s1); ++m) {
            if (m >= m0 && m < m1) floor_point(m);
            if (m >= s0 && m < s1) slab_point(m);
        }
        return;
    }
    for (uint32_t m = m0; m < m1; ++m) floor_point(m);
    if (!slab) return;
    visible_points(h2, h1, za, zb, s.nz, s0, s1);
    for (uint32_t m = s0; m < s1; ++m) slab_point(m);
}

__global__ void k_scatter_resolve(const RenderParams p, const ScatterParams s) {
    const CamDev &c = p.cams[blockIdx.y];
    const uint32_t n = c.w * c.h;
    const uint32_t pix = blockIdx.x * blockDim.x + threadIdx.x;
    if (pix >= n) return;
    const uint32_t word = c.hit_cell[pix];
    if (word == kEmpty) {
        if (c.layer) c.layer[pix] = 255;
        if (c.face) c.face[pix] = kFaceMiss;
        if (c.depth) c.depth[pix] = __int_as_float(0x7f800000);
        if (c.rgba) c.rgba[pix] = kSkyColour;
        return;
    }
    const float depth = __fmul_rn((float)(word >> 8), s.per_step);
    const int32_t px = (int32_t)(pix % c.w), py = (int32_t)(pix / c.w);
    const int32_t a = 2 * px + 1 - (int32_t)c.w, b = (int32_t)c.h - 1 - 2 * py;
    const float dx = (float)(c.F[0] + a * c.R[0] + b * c.U[0]);
    const float dy = (float)(c.F[1] + a * c.R[1] + b * c.U[1]);
    const float dz = (float)(c.F[2] + a * c.R[2] + b * c.U[2]);
    const float dl = __fsqrt_rn(dot3(dx, dy, dz, dx, dy, dz));
    const float kk = __fdiv_rn(depth, dl);
    const float ox = __fmul_rn(__int2float_rn(c.o[0]), 1.0f / 65536.0f);
    const float oy = __fmul_rn(__int2float_rn(c.o[1]), 1.0f / 65536.0f);
    const float xw = __fadd_rn(ox, __fmul_rn(dx, kk)), yw = __fadd_rn(oy, __fmul_rn(dy, kk));
    const float cx = fminf(fmaxf(floorf(xw), 0.0f), (float)(p.world.W - 1));
    const float cy = fminf(fmaxf(floorf(yw), 0.0f), (float)(p.world.H - 1));
    c.hit_cell[pix] = (uint32_t)cy * (uint32_t)p.world.W + (uint32_t)cx;
    if (c.layer) c.layer[pix] = (uint8_t)((word >> 3) & 1);
    if (c.face) c.face[pix] = kFacePZ;
    if (c.depth) c.depth[pix] = depth;
    if (c.rgba) c.rgba[pix] = s.colour[word & 7];
}

}  // namespace

int launch_scatter(const RenderParams &p, const ScatterParams &s, uint32_t n_cams, int sm_count,
                   void *stream) {
    cudaStream_t st = (cudaStream_t)stream;
    const uint32_t px_blocks = (s.max_pixels + kScatterThreads - 1) / kScatterThreads;
    k_scatter_clear<<<dim3(px_blocks < 1024 ? px_blocks : 1024, n_cams), kScatterThreads, 0, st>>>(p);
    const dim3 grid((s.nu * s.nv + kScatterThreads - 1) / kScatterThreads, n_cams);
    // four of the eight blocks that an SM holds: 256 x 256 samples of one view are
    // 1.7 (FEW 10 % faster with 32 points), 512 x 512 6.7 (1 % slower)
    if (grid.x * n_cams <= 4 * (uint32_t)sm_count)
        k_scatter<true><<<grid, kScatterThreads, 0, st>>>(p, s);
    else
        k_scatter<false><<<grid, kScatterThreads, 0, st>>>(p, s);
    if (!s.raw)
        k_scatter_resolve<<<dim3(px_blocks, n_cams), kScatterThreads, 0, st>>>(p, s);
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

}  // namespace hf
