"""How small work is spread over the GPU, read off the plan of random expressions whose results the parity tests compare: a few
outputs with long sums are no single block, many short sums leave no lane idle, and long serial chains go to the interpreter."""
import re

import pytest

from paper_1711_01348_b200 import Plan
from workloads.random_expr import random_expression


@pytest.mark.parametrize("level,seed", [(3, 9), (3, 17), (3, 26), (3, 38), (3, 49)])
def test_long_terms_are_shared_out(level, seed):
    e = random_expression(seed, level)
    plan = Plan(e)
    for q in range(len(e.accesses)):
        for outputs, terms, shares in re.findall(r"; point program: (\d+) outputs x (\d+) terms.*, (\d+) shares", plan.disassemble(q)):
            assert int(outputs) > 4 or int(terms) < 2000 or int(shares) > 1


def test_many_short_sums_leave_no_lane_idle():
    text = Plan(random_expression(32, 4)).disassemble(-1)
    assert re.search(r"277440 outputs x 12 terms.* 1 lanes per output", text)


@pytest.mark.parametrize("level,seed", [(3, 40), (3, 41), (3, 42)])
def test_serial_chains_are_interpreted(level, seed):
    assert "; point program" not in Plan(random_expression(seed, level)).disassemble(-1)
