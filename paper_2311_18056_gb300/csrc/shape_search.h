// The search for a kernel's fastest launch shape, without the launches.
#pragma once

#include <algorithm>

namespace rq {

// Times shapes 0 .. shapes - 1 of a family, in whose order the time falls, if at all, to one
// minimum and then rises: it ends at the first shape 1.3x slower than its best, or 3x slower
// than *best, the least so far of all families.  time(k, warm, &ms) makes a short run of shape
// k (warm, ms < 0: the shape is not possible) or the run that counts, and returns an error code.
// *best and *chosen are updated if a shape beats *best.
//
// A run is late now and then, by any amount: one late run must not end a family, and with it keep
// a worse shape for the handle's life.  So a shape that looks slow is given up only if its short
// run, beside the family's others, was slow as well; else the run that counts is made again.
// (Shapes within their own spread of each other are still told apart by one run: at n = m = 640
// 64 CTAs take 69 to 80 us for 25 layers and 128 CTAs 65 to 95, and of 20 set-ups up to 5 keep
// 128 or 152 CTAs, 12 to 17 % slower over a whole solve.)
template <class Time>
inline int search_family(int shapes, Time time, float* best, int* chosen) {
    float family = 1e30f, family_warm = 1e30f;
    for (int k = 0; k < shapes; ++k) {
        float warm = 0.f, ms = 0.f;
        if (const int rc = time(k, true, &warm)) return rc;
        if (warm < 0.f) continue;
        if (const int rc = time(k, false, &ms)) return rc;
        const float bound = std::min(1.3f * family, 3.0f * *best);
        if (ms > bound && warm <= 1.3f * family_warm) {
            float again = 0.f;
            if (const int rc = time(k, false, &again)) return rc;
            ms = std::min(ms, again);
        }
        if (ms > bound) break;
        family = std::min(family, ms);
        family_warm = std::min(family_warm, warm);
        if (ms < *best) {
            *best = ms;
            *chosen = k;
        }
    }
    return 0;
}

}  // namespace rq
