"""The bench names the kernels that ran and measures the resident loops
against the instruction issue that bounds them."""
import os
import sys

import pytest

import workloads as W

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
import bench  # noqa: E402


def test_issue_roofline_of_the_survey_grid():
    # 59 packed operations per four nodes, two cycles each: 118 cycles per row of 128 nodes on a scheduler, so 608
    # schedulers at 2070 MHz take 1.54 us for one field's level
    rows = W.SURVEY_2D.npad / 128
    floor = rows * 118 / (152 * 4) / 2070e6
    assert floor == pytest.approx(1.54e-6, rel=0.01)
    r = bench.issue_roofline(W.SURVEY_2D.npad, 1, 2 * floor, 152, 2070.0)
    assert r["frac"] == pytest.approx(0.5) and r["bound"] == "fp32 issue"
    assert bench.issue_roofline(W.SURVEY_2D.npad, 2, 2 * floor, 152, 2070.0)["frac"] == pytest.approx(1.0)


def test_loops_are_told_from_their_launches():
    # per shot of 12 500 steps: both resident (in parts), both by steps, two levels per forward launch with a resident
    # reverse loop, and a reverse loop alone by steps
    nt = 12500
    for per_shot, want in ((6 + 23 + 45, (True, True)), (6 + 2 * nt + 1, (False, False)), (6 + nt // 2 + 45, (False, True)),
                           (6 + 23 + nt + 1, (True, False)), (6 + nt // 2 + nt + 1, (False, False))):
        assert bench.resident_loops(8 * per_shot, 8, nt) == want
    assert bench.resident_loops(7, 1, 20) == (True, True)   # a short record: nothing but the shot's own launches


def test_traffic_covers_every_source_of_the_loops():
    assert set(bench._SRC2) >= {"rbc_resident.cu", "rbc_resident.cuh", "rbc_tile2d.cuh", "rbc_stencil.cuh", "rbc_internal.cuh"}
