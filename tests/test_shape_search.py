"""The launch-shape search (csrc/shape_search.h) on given times, compiled for the host: a late run neither ends a
family nor costs more than itself, a family ends where exact times end it, and of close shapes the one that is
faster in the long run is chosen."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.abspath(__file__)), "..", "paper_2311_18056_gb300", "csrc")

# argv: best so far, then per shape the times of its short run and its runs "a,b,.." (the last one again from then on;
# -1: not possible, -2: error); or "random", a number of searches, and per shape least, most (uniform)
MAIN = r"""
#include "shape_search.h"
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <random>
struct S { std::vector<float> t; size_t runs; };
static std::vector<float> list(const char* a) {
    std::vector<float> v;
    for (char* p = const_cast<char*>(a); *p;) {
        v.push_back(std::strtof(p, &p));
        if (*p == ',') ++p;
    }
    return v;
}
int main(int argc, char** argv) {
    std::vector<S> s;
    if (!std::strcmp(argv[1], "random")) {
        for (int i = 3; i < argc; ++i) s.push_back({list(argv[i]), 0});
        std::mt19937 gen(7);
        std::vector<int> won(s.size());
        long runs = 0;
        for (int n = std::atoi(argv[2]); n > 0; --n) {
            float best = 1e30f;
            int chosen = -1;
            auto time = [&](int k, bool warm, float* ms) {
                const float u = (gen() >> 8) * (1.0f / 16777216.0f);
                *ms = (s[k].t[0] + u * (s[k].t[1] - s[k].t[0])) * (warm ? 0.25f : 1.0f);
                runs += !warm;
                return 0;
            };
            std::vector<rq::ShapeTime> timed;
            if (rq::search_family((int)s.size(), time, &best, timed) || rq::pick_shape(timed, time, &chosen)) return 3;
            ++won[chosen];
        }
        for (int w : won) std::printf("%d ", w);
        std::printf("%ld\n", runs);
        return 0;
    }
    for (int i = 2; i < argc; ++i) s.push_back({list(argv[i]), 0});
    float best = std::atof(argv[1]);
    int chosen = -1, runs = 0;
    auto time = [&](int k, bool warm, float* ms) {
        if (s[k].t[0] == -2.f) return -7;
        *ms = s[k].t[warm ? 0 : std::min(++s[k].runs, s[k].t.size() - 1)];
        runs += !warm;
        return 0;
    };
    std::vector<rq::ShapeTime> timed;
    int rc = rq::search_family((int)s.size(), time, &best, timed);
    const int searched = runs;
    if (rc == 0) rc = rq::pick_shape(timed, time, &chosen);
    std::printf("%d %d %d %d\n", rc, chosen, searched, runs);
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("shape")
    (d / "main.cpp").write_text(MAIN)
    subprocess.run([cxx, "-std=c++17", "-O1", "-I", CSRC, "-o", str(d / "main"), str(d / "main.cpp")], check=True)

    def run(args):
        out = subprocess.run([str(d / "main")] + args, check=True, capture_output=True, text=True).stdout
        return tuple(int(v) for v in out.split())

    return run


@pytest.fixture(scope="module")
def search(program):
    def run(shapes, best=1e30):
        """shapes: a time, or (short run, run, ..); a short run takes a fifth and 4 more.  Error, shape, runs of the
        search, all runs."""
        return program(["%g" % best] + [",".join("%g" % t for t in (s if isinstance(s, tuple) else (s / 5 + 4 if s > 0 else s, s)))
                                        for s in shapes])

    return run


@pytest.mark.parametrize("k,late", [(k, late) for k in range(3) for late in (1.2, 1.5, 5.0, 1000.0)] + [(3, 1.2), (3, 5.0), (3, 1000.0)])
def test_a_late_run_does_not_end_a_family(search, k, late):
    times = [100.0, 80.0, 60.0, 50.0, 90.0]
    shapes = list(times)
    shapes[k] = (times[k] / 5 + 4, late * times[k], times[k])
    assert search(shapes)[:2] == (0, 3)
    # a late short run (a kernel's first launch, say) only leaves the decision to the others
    shapes[k] = (late * (times[k] / 5 + 4), times[k])
    assert search(shapes)[:2] == (0, 3)


def test_a_family_ends_where_exact_times_end_it(search):
    # one run each; 120 is 1.5x the best, in its short run too; 50 is not reached; nothing is close to 80
    assert search([110, 80, 101, 120, 50]) == (0, 1, 4, 4)
    # 2x slower than the best of the families before, short runs unknown there: a second run
    assert search([400, 100], best=120.0) == (0, -1, 2, 2)
    assert search([230, 110], best=120.0) == (0, 1, 2, 2)


def test_close_shapes_are_run_again(search):
    assert search([91, 80]) == (0, 1, 2, 4)       # out after two runs
    assert search([84, 80]) == (0, 1, 2, 6)       # never: three runs each
    assert search([81, 80]) == (0, 1, 2, 4)       # within 3 % after two: either will do


def test_uneven_shapes_do_not_win_by_early_runs(program):
    # as measured at n = m = 640, with a slower shape before and after: 152, 128, 64 and 32 CTAs
    *won, runs = program(["random", "2000", "134,160", "126,164", "123,135", "156,161"])
    assert won[2] >= 1940, won
    assert runs <= 2000 * 10


def test_impossible_shapes_and_errors(search):
    assert search([-1, 90, -1, 60]) == (0, 3, 2, 2)
    assert search([-1]) == (0, -1, 0, 0)
    assert search([70, -2])[0] == -7
