"""Launches per step that bench.py reports for solvers that launch their stages one by one: the limits are those of the
sources, and both sides of each."""
import os
import re

import bench
import pytest


def test_limits_are_those_of_the_sources():
    text = "".join(open(os.path.join(bench.ROOT, "paper_2211_16933_gb300", "csrc", f), encoding="utf-8").read()
                   for f in ("qlbm_api.cu", "qlbm_internal.h"))
    for name, value in (("kCellChunk", bench.CELL_CHUNK), ("kNarrowCells", bench.NARROW_CELLS),
                        ("kNarrowCellsQ8", bench.NARROW_CELLS_Q8), ("kCellBall", bench.CELL_BALL),
                        ("kNarrowBall", bench.NARROW_BALL)):
        assert int(re.search(rf"\b{name} = (\d+)", text).group(1)) == value


@pytest.mark.parametrize("fp64,Q,nx,ball,want", [
    (True, 32, 131072, None, 6), (True, 32, 131073, None, 3), (True, 32, 131073, 2, 6), (True, 32, 640, 5, 6),
    (True, 32, 640, 6, 12), (True, 200, 131073, None, 12), (False, 32, 16384, None, 3), (False, 32, 16385, 2, 6),
    (False, 8, 13680, None, 3), (False, 8, 13681, 3, 3), (False, 16, 100, 16, 3), (False, 16, 100, 17, 6)])
def test_launches_per_step(fp64, Q, nx, ball, want):
    kern, launches = bench._step_kernels(fp64, Q, nx, ball)
    assert launches == want
    assert ("narrow" in kern) == (not fp64 and launches == 3)
