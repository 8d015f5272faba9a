"""The launch-shape search (csrc/shape_search.h) on given times, compiled for the host: a late run neither ends a
family nor costs more than itself, and a family ends where exact times end it."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.abspath(__file__)), "..", "paper_2311_18056_gb300", "csrc")

# argv: best so far, then per shape "short run,run,run" (-1: not possible, -2: error)
MAIN = r"""
#include "shape_search.h"
#include <cstdio>
#include <cstdlib>
#include <vector>
int main(int argc, char** argv) {
    struct S { float t[3]; int runs; };
    std::vector<S> s;
    for (int i = 2; i < argc; ++i) {
        S v{};
        if (std::sscanf(argv[i], "%f,%f,%f", v.t, v.t + 1, v.t + 2) != 3) return 2;
        s.push_back(v);
    }
    float best = std::atof(argv[1]);
    int chosen = -1, runs = 0;
    const int rc = rq::search_family((int)s.size(), [&](int k, bool warm, float* ms) {
        if (s[k].t[0] == -2.f) return -7;
        *ms = s[k].t[warm ? 0 : ++s[k].runs];
        runs += !warm;
        return 0;
    }, &best, &chosen);
    std::printf("%d %d %g %d\n", rc, chosen, best, runs);
}
"""


@pytest.fixture(scope="module")
def search(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("shape")
    (d / "main.cpp").write_text(MAIN)
    subprocess.run([cxx, "-std=c++17", "-O1", "-I", CSRC, "-o", str(d / "main"), str(d / "main.cpp")], check=True)

    def run(shapes, best=1e30):
        """shapes: a time, or (short run, run, run); a short run takes a fifth and 4 more."""
        args = [",".join("%g" % t for t in (s if isinstance(s, tuple) else (s / 5 + 4 if s > 0 else s, s, s)))
                for s in shapes]
        out = subprocess.run([str(d / "main"), "%g" % best] + args, check=True, capture_output=True, text=True).stdout
        rc, chosen, got, runs = out.split()
        return int(rc), int(chosen), float(got), int(runs)

    return run


@pytest.mark.parametrize("k,late", [(k, late) for k in range(3) for late in (1.2, 1.5, 5.0, 1000.0)] + [(3, 5.0), (3, 1000.0)])
def test_a_late_run_does_not_end_a_family(search, k, late):
    times = [100.0, 80.0, 60.0, 50.0, 90.0]
    shapes = list(times)
    shapes[k] = (times[k] / 5 + 4, late * times[k], times[k])
    assert search(shapes)[:3] == (0, 3, 50.0)
    # a late short run (a kernel's first launch, say) only leaves the decision to the others
    shapes[k] = (late * (times[k] / 5 + 4), times[k], times[k])
    assert search(shapes)[:3] == (0, 3, 50.0)


def test_a_family_ends_where_exact_times_end_it(search):
    # one run each; 120 is 1.5x the best, in its short run too; 50 is not reached
    assert search([100, 80, 90, 120, 50]) == (0, 1, 80.0, 4)
    # 3x slower than the best of the families before, short runs unknown there: a second run
    assert search([400, 100], best=120.0) == (0, -1, 120.0, 2)
    assert search([300, 110], best=120.0) == (0, 1, 110.0, 2)


def test_impossible_shapes_and_errors(search):
    assert search([-1, 70, -1, 60]) == (0, 3, 60.0, 2)
    assert search([-1]) == (0, -1, 1e30, 0)
    assert search([70, -2])[0] == -7
