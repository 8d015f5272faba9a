"""The tile rule of the FP32 batch products (csrc/tile32.h), compiled for the host, on measured layers: the chosen tile
is close to the best one from the smallest to the largest launches."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.abspath(__file__)), "..", "paper_2311_18056_gb300", "csrc")

MAIN = r"""
#include "tile32.h"
#include <cstdio>
#include <cstdlib>
int main(int argc, char** argv) {
    for (int i = 1; i + 2 < argc; i += 3) {
        const rq::Tile32 t = rq::tile32(std::atoi(argv[i]), std::atoi(argv[i + 1]), std::atoi(argv[i + 2]), 152);
        std::printf("%d %d\n", t.ts, t.tr);
    }
}
"""

# n + m, QPs (one bank group), us per layer in tiles of 32 x 32, 64 x 32 and 64 x 64 on one GB300
MEASURED = [
    (520, 32, 14.5, 17.9, 30.5),
    (520, 200, 19.6, 20.6, 35.9),
    (520, 1000, 40.8, 39.3, 35.8),
    (720, 300, 27.3, 25.5, 43.9),
    (1000, 64, 22.5, 31.5, 55.1),
    (1000, 300, 51.3, 56.4, 65.0),
    (1000, 1000, 127.5, 114.6, 81.3),
    (1300, 128, 42.2, 39.6, 68.5),
    (1300, 200, 45.5, 68.9, 80.5),
    (1300, 500, 122.3, 108.4, 102.1),
    (1600, 32, 33.7, 42.8, 74.1),
    (1600, 200, 97.3, 82.5, 97.0),
    (1600, 700, 197.3, 170.8, 119.5),
    (2300, 50, 69.9, 62.8, 109.8),
    (2300, 128, 73.7, 63.3, 110.5),
    (2300, 160, 139.5, 119.7, 133.9),
    (2300, 500, 279.6, 241.9, 167.6),
    (2300, 1000, 548.3, 482.5, 329.8),
    (3200, 96, 100.8, 160.3, 180.3),
    (3200, 128, 191.0, 162.7, 138.0),
    (3200, 384, 386.9, 328.4, 227.8),
    (3200, 1000, 1037.9, 890.1, 658.1),
]


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("tile")
    (d / "main.cpp").write_text(MAIN)
    subprocess.run([cxx, "-std=c++17", "-O1", "-I", CSRC, "-o", str(d / "main"), str(d / "main.cpp")], check=True)

    def run(cases):
        args = [str(v) for c in cases for v in c]
        out = subprocess.run([str(d / "main")] + args, check=True, capture_output=True, text=True).stdout
        return [tuple(int(v) for v in line.split()) for line in out.splitlines()]

    return run


def test_chosen_tile_is_close_to_the_best(rule):
    tiles = [(32, 32), (64, 32), (64, 64)]
    loss = []
    for (rows, active, *us), tile in zip(MEASURED, rule([(r, b, 1) for r, b, *_ in MEASURED])):
        loss.append(us[tiles.index(tile)] / min(us))
        assert loss[-1] <= 1.2, (rows, active, tile, us)
    assert sum(loss) / len(loss) <= 1.04


def test_every_size_has_a_tile(rule):
    cases = [(r, b, nr) for r in (1, 31, 513, 40000) for b in (1, 33, 1 << 20) for nr in (1, 16)]
    assert all(t in ((32, 32), (64, 32), (64, 64)) for t in rule(cases))
