// Tile (slots x rows) of an FP32 batch product: the rule, without the launches.
#pragma once

#include <algorithm>
#include <cmath>

namespace rq {

struct Tile32 {
    int ts, tr;
};

// Time of a launch per 64 columns of k, us, with c CTAs per SM on average.  Two CTAs of 32 x 32
// share an SM and hide each other's latency (2.0 for two; one on each SM would take 1.25, but the
// SMs that still hold a CTA of the layer before leave some of the others with two); a CTA of
// 64 x 32 takes 1.65 whatever runs beside it; two of 64 x 64 4.5, one 2.9 to 3.7.
inline double tile32_time(Tile32 t, double c) {
    const double k = std::ceil(c), pairs = std::floor(c / 2), rest = c - 2 * pairs;
    if (t.ts == 32) return 2.0 * pairs + (rest <= 0.0 ? 0.0 : rest < 1.0 ? 1.25 + 0.75 * rest : 2.0);
    if (t.tr == 32) return std::max(1.75, 1.65 * k);
    return 4.5 * std::floor(k / 2) + (std::fmod(k, 2.0) == 0.0 ? 0.0 : k == 1.0 ? 2.9 + 0.8 * c : 3.0);
}

// The tile of least time for `rows` rows and `active` QPs in up to nr bank groups, each with a part
// of a tile left over.  Over 98 sizes (n + m = 520 to 3200, 12 to 1000 QPs) 1.0 % slower on average
// than the best tile of each, at most 18 %; with all CTAs of an SM taken to share its FMAs alone it
// was 7 % and 79 % (n + m = 2300, 128 QPs: 109 us a layer in tiles of 64 x 64, 63 in 64 x 32).
inline Tile32 tile32(int rows, int active, int nr, int sms) {
    Tile32 best{32, 32};
    double best_t = 1e300;
    for (const Tile32 c : {Tile32{64, 64}, Tile32{64, 32}, Tile32{32, 32}}) {
        const double slots = (active + c.ts - 1) / c.ts + (active > c.ts ? 0.5 * (nr - 1) : 0.0);
        const double t = tile32_time(c, (rows + c.tr - 1) / c.tr * slots / sms);
        if (t < best_t) {
            best_t = t;
            best = c;
        }
    }
    return best;
}

}  // namespace rq
