// lf_post_plan.h -- how the post-filter divides its views into chunks of rows (host
// arithmetic only).
#pragma once

#include <stdint.h>

namespace lfk {

// One view: strips of columns, and bands of rows of a chunk's smallest length.
struct PostExtent {
    uint64_t strips, bands;
};

inline uint64_t post_ctas(const PostExtent *v, uint32_t n_views, uint64_t chunk)
{
    uint64_t ctas = 0;
    for (uint32_t k = 0; k < n_views; ++k) ctas += v[k].strips * ((v[k].bands + chunk - 1) / chunk);
    return ctas;
}

// Bands per chunk: the length that takes the fewest steps. A wave of the resident
// slots costs its chunk's bands, one more for the six rows before it and about as
// much again to start its CTAs, so the candidates are the shortest chunks that fit
// the fewest waves the strips leave possible, and one, two and three waves more
// (more would save little: 6% for 20 views of 1920 x 1080). Those 20 views have 320
// strips, two waves of 304 slots at least, and run in 45-band chunks (5 waves): 1.41
// ms; in 180-band ones, the second of 2 waves nearly empty, 2.07. 32 views of
// 1440 x 1600: 2.35 ms instead of 3.11.
inline uint64_t post_chunk_bands(const PostExtent *v, uint32_t n_views, uint64_t slots)
{
    uint64_t strips = 0, longest = 1;
    for (uint32_t k = 0; k < n_views; ++k) {
        strips += v[k].strips;
        longest = v[k].bands > longest ? v[k].bands : longest;
    }
    const uint64_t least = strips > slots ? (strips + slots - 1) / slots : 1;
    uint64_t chunk = longest;
    double best = 1e300;
    for (uint64_t waves = least; waves < least + 4; ++waves) {
        uint64_t lo = 1, hi = longest;                   // a chunk of the longest view's bands fits
        while (lo < hi) {
            const uint64_t mid = (lo + hi) / 2;
            if (post_ctas(v, n_views, mid) <= waves * slots) hi = mid; else lo = mid + 1;
        }
        const double steps = (double)waves * ((double)lo + 2.3);
        if (steps < best) {
            best = steps;
            chunk = lo;
        }
        if (lo == 1) break;
    }
    return chunk;
}

}  // namespace lfk
