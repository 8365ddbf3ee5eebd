// hf_rules.h -- how a render is launched, by its cameras (host code).
#pragma once

#include <cstdint>

#include "hf.h"

namespace hf {

// A beam pays where the rays of a warp go through the same cells.  The angle that
// the warp's group of 32 pixels spans (8 x 4, or a row of a wide tile), times the
// length of the world, says how far they fall apart.  Rays each by itself over
// beams, single views and batches of 16, with and without shadows, 8 x 4 tiles:
//   span (rad)   0.017        0.025       0.033       0.05        0.067       0.1
//   256^2        1.29 - 1.85  1.28 - 1.8  1.07 - 1.7  1.01 - 1.65 0.91 - 1.43 0.77 - 1.48
//   2048^2       1.47 - 1.80  1.28 - 1.8  1.11 - 1.4  0.90 - 1.73 0.78 - 1.60 0.66 - 1.73
//   2048 x 8192  1.49 - 2.03  1.16 - 1.9  0.73 - 2.0  0.21 - 1.54 0.17 - 1.48 0.12 - 1.39
// So spans up to 0.04 get beams, up to 0.06 in worlds of up to 512 cells, and up to
// 0.028 in worlds of more than 4096.
inline bool view_wide(int32_t W, int32_t H, const hf_camera &k, uint32_t tw) {
    const int32_t size = W > H ? W : H;
    const double most = size <= 512 ? 0.06 : size <= 4096 ? 0.04 : 0.028;
    const double gw = tw < 32 ? tw : 32, gh = 32 / gw;
    auto norm2 = [](const int32_t *v) {
        return (double)v[0] * v[0] + (double)v[1] * v[1] + (double)v[2] * v[2];
    };
    // neighbouring pixels are 2 |right|, 2 |up| apart at distance |fwd|
    const double across = 4.0 * gw * gw * norm2(k.right), along = 4.0 * gh * gh * norm2(k.up);
    return (across > along ? across : along) > most * most * norm2(k.fwd);
}

// Whether a batch takes the kernel with beams: if of `share` pixels at most one is a
// wide view's (wide: where to say which views are).  In a batch that does, the rays of
// its wide views go each by itself too (CamDev::single; in beams, batches over 2048 x
// 16384 cells with 3 % of their pixels in views of 64 x 48 took up to seven times as
// long), but in a kernel whose registers are the beams'.  All rays by themselves over
// beams for the views that fit, by the share of the wide views' pixels:
//   share           0.08         0.13         0.21         0.37         0.57         0.84
//   traced, 2048^2  0.99 - 1.59  1.17 - 1.49  1.23 - 1.55  1.09 - 1.42  0.91 - 1.22  0.95 - 1.20
//   2048 x 16384    1.34 - 1.71  1.33 - 1.51  1.33 - 1.63  1.13 - 1.27  0.91 - 1.14  0.86 - 1.00
//   (32 views of 320 x 200 and 64 of 200 x 150, a quarter to half of them wide, the six
//   that lose most: 0.84 - 0.95; so the line is at a quarter)
//   share           0.04         0.07         0.17         0.20         0.44         0.55
//   marched, 100    0.86 - 1.78  0.98 - 1.30  0.85 - 1.32  1.00 - 1.25  0.81 - 1.06  0.94 - 1.00
//   samples; 256    1.26 - 2.97  0.76 - 1.64  1.00 - 2.04  0.77 - 1.58  1.00 - 1.48  1.00 - 1.37
constexpr uint32_t kTraceShare = 4, kMarchShare = 32;
inline bool beams_fit(int32_t W, int32_t H, const hf_camera *cams, uint32_t n, uint32_t tw,
                      uint32_t share, uint8_t *wide) {
    uint64_t all = 0, some = 0;
    for (uint32_t i = 0; i < n; ++i) {
        const uint64_t px = (uint64_t)cams[i].w * cams[i].h;
        wide[i] = view_wide(W, H, cams[i], tw);
        all += px;
        if (wide[i]) some += px;
    }
    return some * share <= all;
}

// Whether a march whose views fit takes beams: from so many samples a ray on that
// can lie in the grid, which is as far as its longer side of the way to the far
// distance.  Below, taking every sample is cheaper: a beam's rounds cost as much
// for few samples.  Every sample over beams, views of 1280 x 800 to 3840 x 2160,
// 2 to 6 of them or one, at the far distance 600, protocol views / near the ground:
//   samples a ray   64                          96                         128
//   protocol        0.70 - 1.44                 0.72 - 1.89                0.73 - 2.30
//   eye level       0.72 - 1.08                 0.80 - 1.33                0.86 - 1.67
// the low ends in worlds of 220 x 300 to 700 x 600 cells.  Over eight sizes of world
// and 64 to 256 samples, beams from 96 samples on lost more than 5 % in 99 of 1232
// renders; from 112 that can lie in the grid, in 27 (cameras near the ground or
// against a wall, whose rays hit at once), for 8 % less in the mean.
inline bool march_beams_pay(int32_t W, int32_t H, int32_t steps, float far_dist) {
    const float size = (float)(W > H ? W : H);
    return (float)steps * (size < far_dist ? size / far_dist : 1.0f) >= 112.0f;
}

// The warp tile of a render that leaves its sides at 0.  8 x 4 is one pixel per
// lane, the most warps: right while a render fills the GPU but a few times over,
// as its slowest warps decide its end.  Beyond that narrow and tall tiles win:
// 32 pixels of 4 x 8 go through nearly the same columns of the grid, and longer
// tiles share one fetch of the tile and of its camera.  Measured over 2048 x 2048
// and 2048 x 16384 cells (us, 8 x 4 against the choice):
//   groups of 32 pixels per resident warp   8 x 4    choice
//   1280 x 720 with shadows       8           81      76  (4 x 8;  4 x 16: 77)
//   960 x 540 with shadows        4           59      61  (4 x 8, so still 8 x 4)
//   1920 x 1080                  15          119     113  (4 x 16; 4 x 8: 118)
//   1920 x 1080 with shadows     18          149     140  (4 x 16; 4 x 32: 142)
//   4K with shadows              71          517     477  (4 x 32; 4 x 16: 487)
//   20 views of 1920 x 1080     355         2142    1952  (4 x 32; 4 x 16: 1997)
// Stores to host memory want wide rows, and the traversal of single rays was
// tuned on 8 x 4: both keep it.
// Tall tiles are for images that fill them: a group of 32 pixels, 8 x 4 or 4 x 8,
// costs a warp the same whether its lanes have pixels or not, and one that has none
// a tenth of it.  So 4 x 8 is taken only if it makes no more groups (batches of
// images of 9 rows: a third more, 185 -> 211 us), and a taller tile only if no more
// than an eighth of its groups are empty.
inline void default_tile(const hf_camera *cams, uint32_t n, bool beams, uint64_t warps,
                         uint32_t flags, uint32_t &tw, uint32_t &th) {
    tw = 8;
    th = 4;
    if (!beams || (flags & HF_HOST_OUTPUTS)) return;
    // groups of 32 pixels; tiles of 8 x 4; groups of 4 x h tiles, h = 8, 16, 32
    uint64_t groups = 0, wide = 0, tall[3] = {0, 0, 0};
    for (uint32_t i = 0; i < n; ++i) {
        const uint64_t w = cams[i].w, h = cams[i].h;
        groups += (w * h + 31) / 32;
        wide += (w + 7) / 8 * ((h + 3) / 4);
        for (int k = 0; k < 3; ++k) tall[k] += (w + 3) / 4 * (((h - 1) >> (3 + k)) + 1) << k;
    }
    if (groups < 6 * warps || tall[0] * 32 > wide * 33 || wide >= 0xFFFFFFFFull) return;
    int k = groups < 12 * warps ? 0 : groups < 64 * warps ? 1 : 2;
    while (k && tall[k] * 8 > tall[0] * 9) --k;
    tw = 4;
    th = 8u << k;
}

}  // namespace hf
