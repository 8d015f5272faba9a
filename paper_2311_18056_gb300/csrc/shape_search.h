// The search for a kernel's fastest launch shape, without the launches.
//
// A run is late now and then, by any amount, and the runs of some shapes differ much more than
// those of others (n = m = 640, 50 layers of the single-QP solve, us: 64 CTAs 123 to 137, 128 CTAs
// 126 to 164 around 146).  With one run each, 5 of 20 set-ups of that size kept 128 or 152 CTAs,
// 12 to 17 % slower over a whole solve, for the handle's life.
#pragma once

#include <algorithm>
#include <vector>

namespace rq {

struct ShapeTime {
    int k;
    float ms;
};

// Times shapes 0 .. shapes - 1 of a family, in whose order the time falls, if at all, to one
// minimum and then rises: it ends at the first shape 1.3x slower than its best, or 2x slower
// than *best, the least so far of all families.  time(k, warm, &ms) makes a short run of shape
// k (warm, ms < 0: the shape is not possible) or the run that counts, and returns an error code.
// The shapes timed are added to `out`.
// A shape that looks slow is given up only if its short run, beside the family's others, was slow
// as well; else the run that counts is made again.
template <class Time>
inline int search_family(int shapes, Time time, float* best, std::vector<ShapeTime>& out) {
    float family = 1e30f, family_warm = 1e30f;
    for (int k = 0; k < shapes; ++k) {
        float warm = 0.f, ms = 0.f;
        if (const int rc = time(k, true, &warm)) return rc;
        if (warm < 0.f) continue;
        if (const int rc = time(k, false, &ms)) return rc;
        const float bound = std::min(1.3f * family, 2.0f * *best);
        if (ms > bound && warm <= 1.3f * family_warm) {
            float again = 0.f;
            if (const int rc = time(k, false, &again)) return rc;
            ms = std::min(ms, again);
        }
        if (ms > bound) break;
        family = std::min(family, ms);
        family_warm = std::min(family_warm, warm);
        *best = std::min(*best, ms);
        out.push_back({k, ms});
    }
    return 0;
}

// Of shapes timed once, the one with the least mean of up to three runs: shapes drop out when their
// mean is 15 or 8 % above the least after one or two runs, and runs end once one is left or all
// are within 3 %.  (A run counts as 1.5x its shape's least at most.)  *chosen = -1: none.
template <class Time>
inline int pick_shape(std::vector<ShapeTime> left, Time time, int* chosen) {
    std::vector<float> lowest;
    for (const ShapeTime& s : left) lowest.push_back(s.ms);
    for (int runs = 1;; ++runs) {
        float least = 1e30f, most = 0.f;
        *chosen = -1;
        for (const ShapeTime& s : left)
            if (s.ms < least) {
                least = s.ms;
                *chosen = s.k;
            }
        if (runs == 3) return 0;
        const float keep = runs == 1 ? 1.15f : 1.08f;
        for (size_t i = left.size(); i-- > 0;) {
            if (left[i].ms <= keep * least) {
                most = std::max(most, left[i].ms);
                continue;
            }
            left.erase(left.begin() + i);
            lowest.erase(lowest.begin() + i);
        }
        if (left.size() < 2 || (runs > 1 && most <= 1.03f * least)) return 0;
        for (size_t i = 0; i < left.size(); ++i) {
            float ms = 0.f;
            if (const int rc = time(left[i].k, false, &ms)) return rc;
            lowest[i] = std::min(lowest[i], ms);
            left[i].ms = (left[i].ms * runs + std::min(ms, 1.5f * lowest[i])) / (runs + 1);
        }
    }
}

}  // namespace rq
