// Which tile and how many K splits the FP32 Gaussian stage A~ = G B (m x s by s x d) takes. Host code only.
#pragma once

#include <stdint.h>

#include <algorithm>

namespace lev {

struct GaussPlan {
    bool wide;          // 128 x 256 tiles, one CTA an SM, else 128 x 128 tiles, two
    int64_t tiles, splits, kchunk;   // tiles of A~, K splits of each, rows of k a split
    // rows of k that the SM with the most CTAs goes through, one wave after the other
    int64_t steps() const { return (tiles * splits + (wide ? 151 : 303)) / (wide ? 152 : 304) * kchunk; }
};

// Split-K: two waves of the wide tile or about four 128 x 128 tiles an SM, which is the same length of an FP32
// chain; at least 256 k a split, 64 where that leaves SMs idle (m = 80, d = 20, s = 1,600: 30 us on 7 CTAs).
inline GaussPlan gauss_plan_of(bool wide, int64_t m, int64_t d, int64_t s) {
    GaussPlan p;
    p.wide = wide;
    p.tiles = (m + 127) / 128 * ((d + (wide ? 255 : 127)) / (wide ? 256 : 128));
    p.splits = wide ? std::max<int64_t>(1, 304 / p.tiles) : (608 + p.tiles - 1) / p.tiles;
    const int64_t per = (s + 255) / 256 * p.tiles >= 152 ? 256 : 64;
    p.splits = std::max<int64_t>(1, std::min(p.splits, (s + per - 1) / per));
    const int64_t step = wide ? 16 : 8;                    // rows of k a stage of shared memory holds
    p.kchunk = ((s + p.splits - 1) / p.splits + step - 1) / step * step;
    return p;
}

// The wide tile (16-byte loads, so d and s multiples of 4) where its steps are no more than the narrow one's: with K
// long a step takes 0.19 to 0.21 us in the wide form and 0.18 to 0.24 in the narrow one (d = 132 to 1,024), and the
// rule names the faster form at 25 shapes of 25. The sketch in ms, narrow and wide: 1024 x 256 x 65536 0.84 and 0.72, 2048 x 512 x
// 32768 1.89 and 1.43, 1040 x 260 x 32768 0.80 both; where the wide tile pads or its second wave is nearly empty
// 768 x 384 x 4096 0.080 and 0.108, 3584 x 896 x 32768 5.52 and 6.17, 2064 x 516 x 32768 2.34 and 2.48.
inline GaussPlan gauss_plan(int64_t m, int64_t d, int64_t s) {
    const GaussPlan narrow = gauss_plan_of(false, m, d, s);
    if (d <= 128 || d % 4 != 0 || s % 4 != 0) return narrow;
    const GaussPlan wide = gauss_plan_of(true, m, d, s);
    return wide.steps() <= narrow.steps() ? wide : narrow;
}

}  // namespace lev
