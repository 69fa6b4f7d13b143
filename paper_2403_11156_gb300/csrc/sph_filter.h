// sph_filter.h -- range and threshold of the density sweep's candidate filter (host code).
//
// The filter compares coordinates in steps of h/512, modulo 2^16, and takes (d/h)^2 in half
// precision (k_density); it may pass too much, but no particle within h may fall out.
//
// A coordinate difference of two particles, in steps, is off by less than one for the rounding to
// whole steps, by one for the carry of the paired addition, and by E for the float rounding of
// (x - origin) 512/h up to |x - origin| = D: 2 particles x 2 roundings x 2^-24 x 512 D/h.  So by
// less than a = 2 + E on each axis.  Beyond 512 steps a half's step is 2, so that an overshoot
// counts twice on the one axis that can have it: over all directions a distance below 512 steps
// comes out below 512 + 2a + a^2/128 (the largest of (512 + 2a - 2t)^2 + (sqrt(1024 t) +
// sqrt(2) a)^2 over 0 <= t <= a, for a up to 80).  The sum of squares rounds three times, by at
// most 2^-11 each between 1 and 2.
//
// D is taken from the scene's origin, as the coordinates are: a domain far from zero is filtered
// like any other: a WCSPH step of 500k particles 50,000 h away takes 281 us as at zero (513 with D
// taken from zero and each rounding counted four times, where every candidate passed).  Scenes up to about 280,000 h long have a threshold below 2 (1.018 up to 100 h,
// 1.03 at 5,000 h, 1.1 at 40,000 h); in longer ones every particle takes the exact test.
#pragma once

#include <cmath>
#include <cstdint>

namespace sph {

struct DensityFilter {
    float scale;       // steps per unit of length
    float reach;       // largest |x - origin| on an axis that it holds for; negative: none
    uint32_t thr;      // threshold on (d/h)^2, a pair of halves (none: minus infinity, nothing passes)
};

// extent: the longest side of the scene's cell grid.  Particles outside are covered up to as far
// again (farther ones take the exact test).
inline DensityFilter density_filter(double h, double extent)
{
    DensityFilter f;
    const double reach = 2.0 * extent + 16.0 * h;
    const double a = 2.0 + 1e-3 + std::ldexp(512.0 * (reach + h) / h, -22);
    const double r = 1.0 + (2.0 * a + a * a / 128.0) / 512.0;
    const double thr = r * r + 2e-3;
    f.scale = (float)(512.0 / h);
    f.reach = thr < 2.0 ? (float)reach : -1.0f;
    // steps of 2^-10 from 1 to 2, rounded up
    const uint32_t half = thr < 2.0 ? 0x3c00u + (uint32_t)std::ceil((thr - 1.0) * 1024.0) : 0xfc00u;
    f.thr = half | half << 16;
    return f;
}

}  // namespace sph
