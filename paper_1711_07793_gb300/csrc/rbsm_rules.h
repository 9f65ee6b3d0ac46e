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

}  // namespace rbsm
