"""Tiles of flat grids (csrc/alb_tiles.h): wide enough that few threads are idle."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2009_13426_gb300", "csrc")

DRIVER = r"""
#include <stdio.h>
#include "alb_tiles.h"
int main() {
  const int blocks[] = {64, 128, 256, 384};
  const int rows[] = {1, 2, 3, 4, 5, 7, 8, 9, 15, 16, 17, 64, 1000, 2147483647};
  for (int b : blocks)
    for (int lg0 = 3; (1 << lg0) <= b; ++lg0)
      for (int ny : rows) printf("%d %d %d %d\n", b, lg0, ny, alb::tile_lg(lg0, b, ny));
}
"""


@pytest.fixture(scope="module")
def shapes(tmp_path_factory):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("tiles")
    (d / "d.cpp").write_text(DRIVER)
    subprocess.run([cxx, "-std=c++17", "-I", CSRC, str(d / "d.cpp"), "-o", str(d / "d")],
                   check=True, capture_output=True, text=True)
    out = subprocess.run([str(d / "d")], check=True, capture_output=True, text=True).stdout
    return [tuple(map(int, line.split())) for line in out.splitlines()]


def test_width_and_height(shapes):
    for block, lg0, ny, lg in shapes:
        assert lg >= lg0 and (1 << lg) <= block  # never narrower, never wider than the block
        height = block >> lg
        assert height >= 1
        assert height < 2 * ny or (1 << (lg + 1)) > block  # at most twice the rows
        if lg > lg0:  # widened only where the rows still fit
            assert (block >> (lg - 1)) >= 2 * ny


@pytest.mark.parametrize("source", ["alb_batch.cu", "alb_kernels.cu"])
def test_single_flows_and_batches_share_the_rule(source):
    with open(os.path.join(CSRC, source)) as f:
        assert "tile_lg(" in f.read()
