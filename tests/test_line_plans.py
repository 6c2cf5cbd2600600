"""Which way a line sum is walked, read off the plan: lanes in step for long ranges, every thread by itself for short ones and
where few positions are elements, whose shares must not be cut."""
import re

import pytest

from paper_1711_01348_b200 import Plan
from tests.test_gpu_lines import CASES


def _line(name, access):
    text = Plan(CASES[name]()).disassemble(access)
    line = next(l for l in text.split("\n") if "; line sums" in l)
    return "in step" in line, int(re.search(r"(\d+) shares", line)[1]), int(re.search(r"(\d+) planes", line)[1])


@pytest.mark.parametrize("name,access,in_step", [
    ("bounds_move_with_the_lane", 1, True), ("two_loops", 1, True), ("stride_5", 0, True),
    ("few_elements", 0, False), ("short_runs", 0, False), ("one_lane_wide", 0, False)])
def test_walk(name, access, in_step):
    got, shares, planes = _line(name, access)
    assert got == in_step
    assert planes == shares
