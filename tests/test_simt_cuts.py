"""How the fp32 engine cuts its units over CTAs (simt_row_parts, simt_step_parts of csrc/lacache_plan.h), against measured times of the
cuts on a B200."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2607_16339_b200", "csrc")
SOURCE = r"""
#include <cstdio>
#include <cstdlib>
#include "lacache_plan.h"
using namespace lacache::plan;
int main(int, char** v) {
  if (v[1][0] == 'b') printf("%d", simt_row_parts(atoll(v[2]), atoi(v[3]), atoi(v[4]), 148));
  else printf("%d", simt_step_parts(atoi(v[3]), atoi(v[4]), atoi(v[2]), atoi(v[5]), atoi(v[6]), 148));
}
"""


@pytest.fixture(scope="module")
def parts(tmp_path_factory):
    d = tmp_path_factory.mktemp("cuts")
    (d / "m.cc").write_text(SOURCE)
    subprocess.run(["g++", "-O1", "-std=c++17", "-I", CSRC, "-I", "/usr/local/cuda/include", str(d / "m.cc"), "-o", str(d / "m")], check=True)
    return lambda *a: int(subprocess.run([str(d / "m")] + [str(x) for x in a], capture_output=True, text=True, check=True).stdout)


# (units, key tiles, features): a build's time in us cut over 1, 2, ... parts
BUILDS = {
    (4, 3, 128): (10.2, 9.0, 9.5),
    (20, 6, 128): (16.0, 13.2, 12.0, 11.7, 13.2, 12.9),
    (48, 7, 64): (14.8, 12.2, 12.7, 11.3, 15.0, 13.8, 12.6),
    (48, 7, 128): (21.4, 16.5, 18.8, 15.3, 19.4, 24.5, 21.6),
    (60, 9, 128): (25.3, 18.6, 19.8, 18.6, 28.2, 28.2, 28.1, 25.8),
    (72, 7, 64): (15.3, 14.9, 14.3, 13.5, 16.9, 21.2, 18.6),
    (80, 8, 128): (23.8, 22.0, 20.7, 24.6, 31.1, 30.4, 34.3, 31.3),
    (96, 5, 128): (18.7, 19.2, 24.3, 23.2, 26.4),
    (96, 14, 128): (36.1, 31.2, 36.3, 34.9, 38.6, 39.8, 42.1, 41.8),
    (108, 4, 128): (15.6, 16.9, 21.0, 21.4),
    (152, 11, 128): (43.5, 36.6, 40.4, 41.3, 49.3, 51.9, 59.3, 61.0),
    (184, 11, 128): (38.3, 42.6, 41.4, 44.3, 52.5, 59.2, 62.6, 66.6),
    (240, 17, 128): (56.8, 63.1, 70.6, 65.2, 87.0, 87.3, 101.3, 90.3),
    (252, 7, 64): (20.9, 27.9, 27.9, 30.6, 40.1, 42.3, 42.1),
    (456, 17, 128): (100.0, 98.2, 115.2, 116.5, 139.4, 156.1, 176.2, 165.2),
    (560, 71, 128): (455.8, 464.9, 512.9, 487.4, 526.5, 535.0, 574.4, 559.7),
    (660, 21, 128): (177.4, 176.9, 200.3, 207.2, 243.5, 258.3, 272.5, 287.7),
    (736, 24, 128): (199.9, 213.1, 243.4, 244.8, 283.6, 297.1, 341.3, 321.3),
}
# (heads, block-row items, fixed-row tiles, key tiles, features): a step's
STEPS = {
    (2, 1, 2, 3, 128): (15.0, 11.6, 8.8),
    (4, 1, 6, 7, 64): (15.4, 11.4, 9.7, 7.6, 8.6, 8.0, 6.7),
    (4, 1, 159, 160, 128): (357.1, 189.5, 137.2, 107.0, 91.9, 97.8, 80.0, 72.6),
    (4, 2, 15, 9, 128): (27.8, 18.2, 14.4, 11.9, 14.1, 14.1, 13.8, 11.8),
    (8, 2, 19, 11, 128): (43.6, 26.1, 20.7, 17.4, 18.4, 16.1, 18.2, 21.0),
    (8, 3, 12, 5, 128): (17.3, 15.3, 12.5, 12.1, 10.8),
    (8, 3, 27, 12, 128): (36.3, 26.1, 21.4, 24.0, 26.7, 25.2, 24.4, 24.5),
    (8, 6, 23, 11, 128): (45.6, 28.6, 35.0, 32.0, 34.1, 31.3, 39.2, 37.9),
    (8, 8, 39, 24, 128): (95.1, 74.3, 70.7, 69.6, 76.4, 75.0, 77.2, 82.1),
    (12, 1, 5, 6, 64): (14.0, 9.8, 8.0, 8.9, 10.1, 8.4),
    (12, 2, 15, 9, 128): (33.7, 23.7, 19.3, 18.1, 22.4, 24.1, 23.6, 22.1),
    (12, 3, 17, 6, 128): (21.1, 15.6, 19.8, 20.4, 21.5, 19.9),
    (12, 3, 55, 21, 128): (79.5, 59.5, 56.9, 53.4, 54.9, 51.9, 58.5, 55.0),
    (12, 6, 38, 17, 128): (77.8, 62.4, 59.6, 59.1, 64.8, 65.1, 69.5, 68.6),
    (16, 2, 97, 51, 64): (121.4, 75.2, 65.5, 59.4, 58.4, 55.6, 56.6, 55.1),
    (32, 4, 51, 14, 128): (118.0, 103.0, 111.4, 111.5, 118.0, 123.5, 124.7, 127.9),
    (40, 1, 9, 10, 128): (43.1, 33.9, 31.5, 34.4, 34.0, 35.9, 37.8, 38.7),
}


@pytest.mark.parametrize("shape", sorted(BUILDS))
def test_cut_of_a_build(parts, shape):
    t = BUILDS[shape]
    assert t[parts("b", *shape) - 1] <= 1.15 * min(t)


@pytest.mark.parametrize("shape", sorted(STEPS))
def test_cut_of_a_step(parts, shape):
    t = STEPS[shape]
    assert t[parts("s", *shape) - 1] <= 1.16 * min(t)


def test_cuts_stay_within_a_cluster(parts):
    for units, tiles in ((1, 1), (200, 1), (1, 3), (100000, 300), (1, 300)):
        assert 1 <= parts("b", units, tiles, 128) <= min(8, tiles)
    for heads, split, rest, tiles in ((1, 1, 0, 1), (64, 16, 400, 1), (64, 16, 400, 200), (1, 1, 0, 200)):
        assert 1 <= parts("s", heads, split, rest, tiles, 64) <= min(8, tiles)
