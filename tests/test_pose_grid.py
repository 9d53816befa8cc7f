"""The general pose's scatter grid (csrc/pose_grid.h) on the host, at frame sizes near the limit
w h < 2^31 that no device test can hold: every column and row has its thread, and the number of
blocks is one launch's."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2506_15183_gb300", "csrc")

PROGRAM = r"""
#include "pose_grid.h"
#include <cstdio>
#include <cstdlib>
int main(int argc, char** argv)
{
    for (int i = 1; i + 1 < argc; i += 2) {
        const yoro::ScatterGrid g = yoro::scatter_grid(atoi(argv[i]), atoi(argv[i + 1]));
        printf("%u %u %d %d\n", g.cols, g.blocks, yoro::kScatterCols, yoro::kScatterRows);
    }
}
"""


@pytest.fixture(scope="module")
def grids(tmp_path_factory):
    d = tmp_path_factory.mktemp("grid")
    (d / "grid.cpp").write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", f"-I{CSRC}", str(d / "grid.cpp"), "-o", str(d / "grid")], check=True)

    def run(*sizes):
        out = subprocess.run([str(d / "grid"), *[str(v) for wh in sizes for v in wh]], check=True, capture_output=True,
                             text=True).stdout
        return [tuple(map(int, line.split())) for line in out.splitlines()]

    return run


def test_blocks_cover_the_frame_once(grids):
    top = 2 ** 31 - 1
    sizes = [(1, 1), (256, 4), (257, 5), (1832, 1920), (top, 1), (top - 255, 1), (top - 254, 1), (1, top), (1, top - 2),
             (257, top // 257), (46340, 46340), (top // 4, 4), (top // 5, 5)]
    for (w, h), (cols, blocks, bc, br) in zip(sizes, grids(*sizes)):
        assert cols == -(-w // bc) and blocks == cols * -(-h // br), (w, h)
        assert blocks <= top  # a launch's grid
