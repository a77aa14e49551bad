// Which tile and how many K splits the FP32 Gaussian stage A~ = G B (m x s by s x d) takes. Host code only.
#pragma once

#include <stdint.h>

#include <algorithm>

namespace lev {

struct GaussPlan {
    bool wide;                       // 128 x 256 tiles, one CTA an SM, else 128 x 128 tiles, two
    int64_t tiles, splits, kchunk;   // tiles of A~, K splits of each, rows of k a split
    double us;                       // estimated time
};

// At least `per` rows of k a split, and no more splits than two waves of the wide tile or about four 128 x 128
// tiles an SM. Time: the waves of CTAs, 0.179 us a row of k for the wide tile, 0.213 for two narrow ones on an SM and
// 0.122 for one alone; the reduction's loop over the splits and the partials' traffic; 8.5 us for the two launches.
// Fitted to 316 shapes (m = 16 to 4,096, d = 8 to 1,024, s = 512 to 65,536, m >= 2 d; three values of `per` in both
// forms): 90% of the estimates are within 9%.
inline GaussPlan gauss_plan_of(bool wide, int64_t per, int64_t m, int64_t d, int64_t s) {
    GaussPlan p;
    p.wide = wide;
    p.tiles = (m + 127) / 128 * ((d + (wide ? 255 : 127)) / (wide ? 256 : 128));
    p.splits = wide ? std::max<int64_t>(1, 304 / p.tiles) : (608 + p.tiles - 1) / p.tiles;
    p.splits = std::max<int64_t>(1, std::min(p.splits, (s + per - 1) / per));
    const int64_t step = wide ? 16 : 8;                    // rows of k a stage of shared memory holds
    p.kchunk = ((s + p.splits - 1) / p.splits + step - 1) / step * step;
    const int64_t ctas = p.tiles * p.splits, rem = ctas % 304;
    const double rows = wide ? 0.179 * (double)((ctas + 151) / 152)
                             : 0.213 * (double)(ctas / 304) + (rem == 0 ? 0.0 : rem <= 152 ? 0.122 : 0.213);
    p.us = 8.5 + rows * (double)p.kchunk + 0.0545 * (double)p.splits + 7.26e-7 * (double)p.splits * (double)m * (double)d;
    return p;
}

// The narrow tile with at least 256 rows a split, unless one with fewer rows (where that leaves SMs idle) is
// estimated at 3% less; the wide tile (16-byte loads, so d and s multiples of 4) where it is estimated at less still.
// Over these shapes the choice is 0.3% slower than the fastest of the six on average, 10% at most. Measured, us, the
// narrow tile with 256 rows a split and the choice: 80 x 20 x 1,600 36 and 17, 40 x 20 x 32,768 45 and 45 (67 with 64
// rows), 128 x 64 x 2,048 41 and 19, 1,024 x 256 x 65,536 793 and 681 (wide), 1,536 x 768 x 1,600 116 and 84 (wide,
// 200 rows), 768 x 384 x 4,096 70 and 73 (wide; 97 with 256 rows), 3,584 x 896 x 32,768 5,444 and 5,444 (6,093 wide).
inline GaussPlan gauss_plan(int64_t m, int64_t d, int64_t s) {
    GaussPlan best = gauss_plan_of(false, 256, m, d, s);
    const double most = 0.97 * best.us;
    for (int64_t per = 128; per >= 64; per /= 2) {
        const GaussPlan p = gauss_plan_of(false, per, m, d, s);
        if (p.us <= most && p.us < best.us) best = p;
    }
    if (d > 128 && d % 4 == 0 && s % 4 == 0)
        for (int64_t per = 256; per >= 64; per /= 2) {
            const GaussPlan p = gauss_plan_of(true, per, m, d, s);
            if (p.us < best.us) best = p;
        }
    return best;
}

}  // namespace lev
