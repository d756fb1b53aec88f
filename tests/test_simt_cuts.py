"""How the fp32 engine cuts its units over CTAs (simt_row_parts, simt_step_parts of csrc/lacache_plan.h with the costs of the kernel
that multiplies on the tensor cores), against measured times of the cuts on a B200."""
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
  if (v[1][0] == 'b') printf("%d", simt_row_parts(atoll(v[2]), atoi(v[3]), atoi(v[4]), 148, SIMT_TENSOR_CORES));
  else printf("%d", simt_step_parts(atoi(v[3]), atoi(v[4]), atoi(v[2]), atoi(v[5]), atoi(v[6]), 148, SIMT_TENSOR_CORES));
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
    (4, 3, 128): (10.5, 8.9, 9.4),
    (20, 6, 128): (16.7, 13.2, 11.7, 11.1, 11.0, 11.4),
    (48, 7, 64): (15.5, 12.7, 13.3, 11.5, 15.2, 14.4, 12.8),
    (48, 7, 128): (21.2, 16.1, 18.3, 15.1, 19.0, 24.0, 21.1),
    (60, 9, 128): (25.5, 18.6, 19.4, 18.5, 27.2, 27.5, 27.5, 25.4),
    (72, 7, 64): (16.1, 12.9, 14.2, 14.6, 16.7, 21.1, 18.4),
    (80, 8, 128): (24.0, 21.9, 20.4, 24.3, 30.4, 29.7, 33.4, 30.6),
    (96, 5, 128): (18.6, 19.2, 24.1, 22.9, 25.8),
    (96, 14, 128): (36.8, 30.8, 36.0, 34.2, 37.7, 38.8, 40.9, 41.0),
    (108, 4, 128): (15.7, 16.8, 20.7, 20.9),
    (152, 11, 128): (43.0, 36.7, 39.7, 40.3, 48.3, 50.5, 57.5, 59.5),
    (184, 11, 128): (37.8, 41.2, 41.1, 43.5, 51.1, 57.4, 61.2, 64.9),
    (240, 17, 128): (56.3, 61.7, 69.7, 63.7, 85.5, 85.1, 99.0, 88.3),
    (252, 7, 64): (21.4, 29.1, 27.4, 31.0, 40.7, 42.4, 42.0),
    (456, 17, 128): (99.1, 96.5, 112.9, 113.7, 137.4, 152.8, 172.8, 161.0),
    (560, 71, 128): (447.2, 454.7, 500.3, 475.9, 515.2, 525.0, 561.6, 547.1),
    (660, 21, 128): (175.2, 172.9, 195.9, 201.4, 238.1, 252.6, 265.3, 281.6),
    (736, 24, 128): (197.5, 208.0, 237.2, 239.3, 277.7, 291.6, 333.6, 314.2),
}
# (heads, block-row items, fixed-row tiles, key tiles, features): a step's
STEPS = {
    (2, 1, 2, 3, 128): (15.4, 13.2, 9.5),
    (4, 1, 6, 7, 64): (16.1, 12.5, 11.2, 8.5, 9.3, 9.0, 7.5),
    (4, 1, 159, 160, 128): (350.3, 187.7, 138.2, 111.6, 94.7, 87.8, 82.7, 78.5),
    (4, 2, 15, 9, 128): (28.1, 18.9, 16.1, 12.3, 14.2, 15.1, 13.9, 11.0),
    (8, 2, 19, 11, 128): (42.5, 27.1, 21.3, 17.4, 18.5, 16.4, 17.9, 20.9),
    (8, 3, 12, 5, 128): (18.2, 15.5, 12.5, 12.1, 10.9),
    (8, 3, 27, 12, 128): (36.8, 26.6, 22.7, 25.3, 28.1, 25.9, 25.3, 25.5),
    (8, 6, 23, 11, 128): (47.2, 30.7, 38.6, 34.8, 37.1, 33.6, 42.7, 40.0),
    (8, 8, 39, 24, 128): (103.0, 85.4, 79.8, 87.3, 96.0, 96.0, 99.3, 100.7),
    (12, 1, 5, 6, 64): (14.9, 11.3, 8.8, 9.4, 11.0, 9.1),
    (12, 2, 15, 9, 128): (34.9, 21.8, 20.4, 17.7, 22.4, 24.2, 23.6, 21.4),
    (12, 3, 17, 6, 128): (20.9, 15.8, 19.8, 20.1, 20.7, 20.0),
    (12, 3, 55, 21, 128): (82.9, 62.8, 60.6, 56.5, 57.1, 54.8, 62.2, 59.1),
    (12, 6, 38, 17, 128): (81.8, 70.2, 67.8, 68.3, 75.0, 75.5, 81.9, 79.3),
    (16, 2, 97, 51, 64): (113.4, 75.0, 65.6, 59.9, 58.0, 55.1, 56.3, 55.1),
    (32, 4, 51, 14, 128): (115.5, 103.6, 111.8, 113.7, 120.1, 127.4, 124.8, 128.1),
    (40, 1, 9, 10, 128): (43.8, 34.4, 32.3, 35.7, 34.8, 37.4, 39.6, 40.9),
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
