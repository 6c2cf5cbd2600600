"""Quotients inside the term of a tile program: a quotient keeps its numerator in Y, so one whose divisor is another quotient of
coupled operands holds three values and must not be taken as a core of two."""
import re

import pytest

from oracle.oracle import max_threads
from paper_1711_01348_b200 import Plan
from workloads import configs as W
from workloads.expr import Builder, unit

PUSH, BINY = 12, 13


def _expr(name, ni, nj, nk, term, sums_j=False):
    """f_ij = sum_k term(x_ik, y_jk, z_ik, w_ik), or f_i, summed over j too"""
    b = Builder(name, [ni] if sums_j else [ni, nj], 2 if sums_j else 1, ["x", "y", "z", "w"], [[ni, nk], [nj, nk], [ni, nk], [ni, nk]])
    i, j, k = unit(3, (0, 1)), unit(3, (1, 1)), unit(3, (2, 1))
    t = term(b, b.load("x", [i, k]), b.load("y", [j, k]), b.load("z", [i, k]), b.load("w", [i, k]))
    s = b.sum(2, 0, nk - 1, t)
    if sums_j:
        b.sum(1, 0, nj - 1, s)
    return b.done()


def _div(b, a, c):
    return b.bin("div", a, c)


TERMS = {
    "x/(y/z)": lambda b, x, y, z, w: b.bin("add", _div(b, x, _div(b, y, z)), w),
    "x/(y/z) alone": lambda b, x, y, z, w: _div(b, x, _div(b, y, b.bin("add", z, w))),
    "w (x/(y/z))": lambda b, x, y, z, w: b.bin("mul", w, _div(b, x, _div(b, y, z))),
    "1/(x/y)": lambda b, x, y, z, w: b.bin("mul", b.bin("add", z, w), _div(b, b.const(1.0), _div(b, x, y))),
    "(x/y)/z": lambda b, x, y, z, w: b.bin("add", _div(b, _div(b, x, y), z), w),
    "(x y)/(z/y)": lambda b, x, y, z, w: b.bin("add", _div(b, b.bin("mul", x, y), _div(b, z, y)), w),
    "x - w/(y/z)": lambda b, x, y, z, w: b.bin("sub", x, _div(b, w, _div(b, y, z))),
    "x/(w - y/z)": lambda b, x, y, z, w: _div(b, x, b.bin("sub", b.bin("add", w, b.const(4.0)), _div(b, y, z))),
}
SIZES = {"columns": (97, 103, 9, False), "summed": (67, 41, 31, True)}


def _case(term, size):
    ni, nj, nk, sums_j = SIZES[size]
    return _expr(term, ni, nj, nk, TERMS[term], sums_j)


@pytest.mark.parametrize("size", sorted(SIZES))
@pytest.mark.parametrize("term", sorted(TERMS))
def test_one_value_waits(term, size):
    e = _case(term, size)
    plan = Plan(e)
    for w in [-1] + [-2 - s for s in range(plan.num_stages())] + list(range(len(e.accesses))):
        for core in re.findall(r"tile program.* core ([0-9a-f]+)", plan.disassemble(w)):
            waits = 0
            for op in (byte & 15 for byte in reversed(bytes.fromhex(core.zfill(16)))):
                waits += (op == PUSH) - (op == BINY)
                assert 0 <= waits <= 1, (w, core)
            assert waits == 0


@pytest.mark.gpu
@pytest.mark.parametrize("size", sorted(SIZES))
@pytest.mark.parametrize("term", sorted(TERMS))
def test_quotients(term, size):
    from tests.gpu_util import check_against_oracle
    e = _case(term, size)
    args, df = W.make_inputs(e, ("uniform", 0.5, 1.5), seed=11)
    check_against_oracle(e, args, df, nthreads=max_threads())
