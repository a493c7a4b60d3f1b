"""Where short lines and the double recovery take tiles (`csrc/tile_plan.h`),
checked on the CPU: a small C++ driver prints the shape of a line, its tiles and
the estimated times, for measured sweeps (GB300, us: tiles, streamed with timed
ranges, streamed untimed) whose two sides lie at least 1.25 apart.  The estimates
must order them alike; before them all of these ran on tiles.  Every line
length's tiles cover it once and none is empty."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1206_0919_gb300", "csrc")

DRIVER = r"""
#include <cstdio>
#include "tile_plan.h"
using namespace shasta;
int main() {
  long long lines;
  int n, axis, rec64;
  while (std::scanf("%lld %d %d %d", &lines, &n, &axis, &rec64) == 4) {
    const int shape = tile_shape_for(n, axis);
    TilePlan t;
    t.shape = shape;
    tile_cut(t, n);
    const SweepCost c = sweep_cost(lines, n, axis, shape, rec64, 152);
    std::printf("%d %d %d %d %g %g %g\n", t.ntile, t.len, tile_own(shape), (int)by_cost(n, rec64), c.tile, c.stream,
                c.untimed);
  }
}
"""

# recovery in double, axis, lines, cells; us on tiles, timed, untimed
MEASURED = [
    (0, 0, 48 * 48, 1, 8.1, 15.2, 261), (0, 0, 48 * 48, 16, 7.0, 21.4, 33.6), (0, 0, 200 * 200, 3, 39.9, 23.4, 112),
    (0, 0, 256 * 256, 5, 60.4, 37.8, 74.8), (0, 0, 256 * 256, 48, 51.6, 72.6, 72.5), (0, 0, 400 * 400, 8, 116, 70.5, 70.1),
    (0, 0, 400 * 400, 16, 115.5, 86.9, 86.9), (0, 0, 512 * 512, 3, 232, 96.3, 133), (0, 0, 1 << 20, 1, 908, 295, 390),
    (0, 0, 1 << 20, 12, 743, 491, 494), (0, 2, 128 * 96, 24, 13.2, 23.2, 23.4), (0, 2, 256 * 256, 1, 56.4, 27.6, 243),
    (0, 2, 400 * 400, 20, 115.5, 88.9, 88.9), (0, 2, 512 * 512, 5, 219, 85.7, 92.7),
    (1, 0, 48 * 48, 256, 98, 176, 182), (1, 0, 128 * 96, 5, 96, 63, 309), (1, 0, 128 * 96, 56, 119, 172, 180),
    (1, 0, 256 * 256, 8, 463, 189, 283), (1, 0, 400 * 400, 16, 1120, 518, 518), (1, 0, 1 << 20, 28, 8553, 4295, 4445),
    (1, 2, 256 * 256, 24, 455, 301, 328), (1, 2, 80 * 80, 128, 121, 175, 178),
]


@pytest.fixture(scope="module")
def driver(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("tp")
    src, exe = d / "tp.cpp", d / "tp"
    src.write_text(DRIVER)
    subprocess.run([cxx, "-O2", "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], check=True)

    def run(rows):
        text = "\n".join("%d %d %d %d" % r for r in rows)
        out = subprocess.run([str(exe)], input=text, capture_output=True, text=True, check=True).stdout
        return [[float(x) for x in ln.split()] for ln in out.splitlines()]
    return run


def test_estimates_order_the_measured_sweeps(driver):
    got = driver([(lines, n, axis, rec64) for rec64, axis, lines, n, *_ in MEASURED])
    for (rec64, axis, lines, n, tile, timed, untimed), r in zip(MEASURED, got):
        assert r[3] == 1
        for k, us in ((5, timed), (6, untimed)):
            if max(us / tile, tile / us) >= 1.25:
                assert (r[4] < r[k]) == (tile < us), (rec64, axis, lines, n, r[4:])


def test_tiles_cover_every_line(driver):
    ns = [n for n in range(1, 700)] + [3069, 10 ** 6 + 1, 2 ** 30]
    for axis in (0, 1):
        for n, (ntile, length, own, *_) in zip(ns, driver([(1000, n, axis, 0) for n in ns])):
            assert 1 <= length <= own and (ntile - 1) * length < n <= ntile * length
