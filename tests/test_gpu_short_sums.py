"""Sums of one to four terms inside an element-wise expression: as terms of a point program up to 50517 outputs, in a thread beyond."""
import pytest

from oracle.oracle import max_threads
from paper_1711_01348_b200 import Plan
from workloads import configs as W
from workloads.expr import Builder, unit


def _tail(n, nk):
    """f_i = tanh(s) + w_i s, s = sum_k sinh(u_ik) log(2 + v_k^2)"""
    b = Builder("tail", [n], 1, ["u", "v", "w"], [[n, nk], [nk], [n]])
    u, v = b.load("u", [unit(2, (0, 1)), unit(2, (1, 1))]), b.load("v", [unit(2, (1, 1))])
    s = b.sum(1, 0, nk - 1, b.bin("mul", b.un("sinh", u), b.un("log", b.bin("add", b.powi(v, 2), b.const(2.0)))))
    b.bin("add", b.un("tanh", s), b.bin("mul", b.load("w", [unit(2, (0, 1))]), s))
    return b.done()


SIZES = [(1, 2), (33, 1), (33, 2), (257, 3), (50517, 3), (50518, 3), (50517, 4)]


@pytest.mark.parametrize("n,nk", SIZES)
def test_taken(n, nk):
    text = Plan(_tail(n, nk)).disassemble(-1)
    spread = nk > 3 or (nk > 1 and n <= 50517)
    assert ("%d outputs x %d terms" % (n, nk if spread else 1)) in text


def _cheap(n, nk):
    """f_i = exp(sum_k u_ik v_k): summands without functions"""
    b = Builder("cheap", [n], 1, ["u", "v"], [[n, nk], [nk]])
    b.un("exp", b.sum(1, 0, nk - 1, b.bin("mul", b.load("u", [unit(2, (0, 1)), unit(2, (1, 1))]), b.load("v", [unit(2, (1, 1))]))))
    return b.done()


# three terms without functions are spread up to 37888 outputs, two up to 50517, four and more up to 75776
CHEAP = [(37888, 3, True), (37889, 3, False), (50517, 2, True), (50518, 2, False), (75776, 4, True)]


@pytest.mark.parametrize("n,nk,spread", CHEAP)
def test_cheap_taken(n, nk, spread):
    assert ("%d outputs x %d terms" % (n, nk if spread else 1)) in Plan(_cheap(n, nk)).disassemble(-1)


@pytest.mark.gpu
@pytest.mark.parametrize("n,nk,spread", CHEAP)
def test_cheap_sums(n, nk, spread):
    from tests.gpu_util import check_against_oracle
    e = _cheap(n, nk)
    check_against_oracle(e, *W.make_inputs(e, ("uniform", -0.9, 0.9), seed=n), nthreads=max_threads())


@pytest.mark.gpu
@pytest.mark.parametrize("n,nk", SIZES)
def test_short_sums(n, nk):
    from tests.gpu_util import check_against_oracle
    e = _tail(n, nk)
    check_against_oracle(e, *W.make_inputs(e, ("uniform", -0.9, 0.9), seed=n), nthreads=max_threads())
