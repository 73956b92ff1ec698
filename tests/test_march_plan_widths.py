"""Host logic of the row march's work items at widths that are no multiple of a strip, and of grids too small to give
every CTA an 8-row item (compiled from the header the library uses; no GPU): strips of one width and a last
one of two columns at least, every node in exactly one item, two rows or more where an item touches a wall,
one wave; a width that no strip fits is refused."""
import os
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1310_7450_gb300", "csrc")
SOURCE = r"""
#include <cstdio>
#include <cstdlib>
#include "lb_march_plan.h"
int main(int, char** v) {
    const int nx = std::atoi(v[1]), ny = std::atoi(v[2]), R = std::atoi(v[3]), nsm = std::atoi(v[4]);
    const int W = lbk::march_strip_width(nx);
    std::printf("%d\n", W);
    if (W == 0 || std::atoi(v[5]) == 0) return 0;
    for (const lbk::MarchItem& i : lbk::short_items(
             lbk::fine_items(lbk::march_plan(nx, ny, R, nsm, lbk::MarchModel{0.08, 1.2, true}), nx, ny, R * nsm), nx))
        std::printf("%d %d %d %d\n", i.x0, i.w, i.y0, i.y1);
}
"""


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    d = tmp_path_factory.mktemp("plan")
    (d / "plan.cpp").write_text(SOURCE)
    exe = str(d / "plan")
    subprocess.run(["g++", "-std=c++17", "-O1", "-Wall", "-Werror", "-I", CSRC, str(d / "plan.cpp"), "-o", exe], check=True)

    def run(nx, ny, R=6, nsm=152, items=True):
        out = subprocess.run([exe, *map(str, (nx, ny, R, nsm, int(items)))], check=True, capture_output=True, text=True).stdout
        lines = out.splitlines()
        return int(lines[0]), np.array([[int(x) for x in l.split()] for l in lines[1:]], dtype=np.int64)
    return run


@pytest.mark.parametrize("nx,ny", [(96, 16), (97, 4300), (100, 60), (129, 3200), (256, 17), (1000, 777), (1001, 777), (8191, 64),
                                   (174721, 16), (200001, 19), (128, 64), (4096, 4096)])
def test_items_cover_every_node_once(plan, nx, ny):
    W, it = plan(nx, ny)
    assert W % 8 == 0 and 8 <= W <= 128
    assert np.all(it[:, 0] % W == 0) and np.all(it[:, 1] == np.minimum(W, nx - it[:, 0])) and it[:, 1].min() >= 2
    assert np.all(it[:, 3] > it[:, 2]) and int(((it[:, 3] - it[:, 2]) * it[:, 1]).sum()) == nx * ny
    strips = -(-nx // W)
    order = np.lexsort((it[:, 2], it[:, 0]))
    s = it[order]
    first = np.r_[True, s[1:, 0] != s[:-1, 0]]
    assert first.sum() == strips and np.all(s[first, 2] == 0)
    assert np.all(s[1:, 2][~first[1:]] == s[:-1, 3][~first[1:]])       # consecutive items of a strip meet
    wall = (it[:, 2] == 0) | (it[:, 3] == ny)
    assert (it[wall, 3] - it[wall, 2]).min() >= 2
    assert len(it) <= max(6 * 152, strips)


def test_items_stay_below_the_range_of_their_offsets(plan):
    _, it = plan(1 << 23, 200)                                         # 65 536 strips: one item each, cut short
    assert ((it[:, 3] - it[:, 2]) << 23).max() <= 1 << 29
    assert int(((it[:, 3] - it[:, 2]) * it[:, 1]).sum()) == 200 << 23


def test_strip_width(plan):
    every = 5765760                                                    # the least common multiple of 8, 16, ... 128
    for nx in (every, every + 2, 720721, 11531519):
        W, _ = plan(nx, 16, items=False)
        assert 8 <= W <= 128 and W % 8 == 0 and nx % W != 1
    for nx in (every + 1, 2 * every + 1):
        assert plan(nx, 16, items=False)[0] == 0
