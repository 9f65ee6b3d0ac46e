// Rules that choose a kernel form by the sizes of a call: host code without
// CUDA, so that they can be tested where there is no GPU.
#pragma once

#include <cstdint>

namespace rbsm {

// Square tiles of `side` texels that cover a width x height map.
inline long long square_tiles(int width, int height, long long side)
{
    return ((width + side - 1) / side) * ((height + side - 1) / side);
}

// The light pass: tiles of kLargeTile texels a side instead of 32.  They need
// the occluders in one culling round (kLightRound of both kinds), and from
// two tiles for each of four CTAs per SM on they are the faster ones where
// there is something to cull and to turn down block by block (one map, us,
// tiles of 64 / of 32, with 24 rectangles and with 140 and 60 spheres:
// 2048^2, below the line, 9.4 / 10.5 and 25.1 / 23.2; 2240^2 10.3 / 11.8 and
// 27.4 / 24.6; 3000^2 14.3 / 18.4 and 33.7 / 34.9; 4096^2 20.4 / 31.4 and
// 53.9 / 56.6; 8192^2 65.2 / 110 and 140 / 179; one rectangle, 4096^2, 16.0 /
// 27.6).  Without occluders a map is its stores, and tiles of 32 make them
// without barriers (4096^2 14.4 / 10.0, 8192^2 51.0 / 43.9).  And with spheres
// and a depth scale outside the float-float range every covered texel takes the
// slow double operations, whose uneven load the small tiles share out better
// (4096^2, 100 rectangles and 50 spheres, 302 / 238).
constexpr int kLargeTile = 64;
constexpr int kLightRound = 256;
inline bool light_large_tiles(int width, int height, int64_t n_rects, int64_t n_spheres, bool scale_in_range, int sms)
{
    const int64_t n = n_rects + n_spheres;
    return n > 0 && n <= kLightRound && (scale_in_range || n_spheres == 0) &&
           square_tiles(width, height, kLargeTile) >= 2LL * 4 * sms;
}

// The light pass with tiles of 32: whether a thread's rows are spread over its
// tile.  From 32 tiles on, up to two for each of four CTAs per SM, the time of
// a map is that of its tiles' slowest warps, and spreading the rows beats turning
// blocks down as a whole (us, spread / blocks, with 24 rectangles, with 140 and
// 60 spheres and with 200 of each: 192^2 3.8 / 4.2, 10.6 / 10.6 and 15.9 / 16.4;
// 256^2 3.5 / 3.6, 8.7 / 9.1 and 13.9 / 15.2; 512^2 3.9 / 4.3, 7.8 / 9.0 and 14.4
// / 15.9; 768^2 4.3 / 4.4, 10.1 / 10.7 and 18.9 / 19.1; 1024^2 5.2 / 5.3, 12.6 / 13.3 and
// 22.4 / 22.9).  On fewer tiles the occluders that fill a block count (128^2 3.8 /
// 4.1, 14.0 / 12.0 and 23.2 / 21.0), and on more the work in all (2048^2 10.3 /
// 10.6, 23.1 / 23.3 and 39.7 / 39.0; with 300 rectangles 41.3 / 38.0, with 200
// large ones 117 / 79).
inline bool light_spread_rows(int width, int height, int sms)
{
    const long long tiles = square_tiles(width, height, 32);
    return tiles > 32 && tiles <= 8LL * sms;
}

// Depth buffers: CTAs of 640 threads (two per SM) where there are 64 tiles of
// 128 pixels for every SM, else of 256 (five per SM), both at 48 registers (us,
// 640 / 256, both answers, with a texture: 320x240 14.0 / 12.1, 4 frames of 1280x720
// 52.5 / 46.4, below the line; 1920x1080 29.2 / 29.4, silhouettes alone 24.9 /
// 26.6, and one frame of 3840x2160 52.7 / 54.7, above).
constexpr int kGbufferLargeThreads = 640, kGbufferSmallThreads = 256;
inline bool gbuffer_large(int width, int height, int sms)
{
    return ((long long)width * height + 127) / 128 >= 64LL * sms;
}

}  // namespace rbsm
