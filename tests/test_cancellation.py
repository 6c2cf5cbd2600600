"""Sums whose summands cancel.  In (a + b)^2 c with a near -b the expanded form c a^2 + 2 c a b + c b^2 loses the digits that
the term as written keeps, so an expression of moderate size, or with a short sum, is evaluated as written: within the
tolerance of every parity test, whose scale is the sum of |terms| of the expression as written."""
import pytest

from oracle.oracle import max_threads
from paper_1711_01348_b200 import Plan
from workloads import configs as W
from workloads.expr import Builder

# index spaces of up to 2^24 elements
MODERATE = [(1000, 1500, 6), (1000, 1000, 16), (4000, 128, 20)]
# larger ones with sums of a few terms
SHORT = [(2500, 2400, 3), (2500, 2400, 5)]


def _offset_inputs(e):
    args, df = W.make_inputs(e, ("uniform", -0.5, 0.5), seed=9)
    args[0] += 30.0
    args[1] -= 30.0
    return args, df


@pytest.mark.parametrize("ni,nj,nk", MODERATE + SHORT)
def test_evaluated_as_written(ni, nj, nk):
    plan = Plan(W.intro(ni, nj, nk))
    for which in [-1] + [-2 - s for s in range(plan.num_stages())]:
        assert "; factored" not in plan.disassemble(which)


@pytest.mark.gpu
@pytest.mark.parametrize("ni,nj,nk", MODERATE + SHORT)
@pytest.mark.parametrize("offset", [True, False])
def test_cancelling_summands(ni, nj, nk, offset):
    from tests.gpu_util import check_against_oracle
    e = W.intro(ni, nj, nk)
    args, df = _offset_inputs(e) if offset else W.make_inputs(e, ("uniform", -0.5, 0.5), seed=nk)
    check_against_oracle(e, args, df, nthreads=max_threads())


def _product(ni, nj, nk):
    """f_i = sum_jk x_ij y_jk: a sum over one product is reordered, not expanded."""
    b = Builder("product", [ni], 2, ["x", "y"], [[ni, nj], [nj, nk]])
    p = b.bin("mul", b.load("x", [[1, 0, 0], [0, 1, 0]]), b.load("y", [[0, 1, 0], [0, 0, 1]]))
    b.sum(1, 0, nj - 1, b.sum(2, 0, nk - 1, p))
    return b.done()


def _all_terms(ni, nj, nk):
    """f_ij = sum_k (w_0 + y_ijk): the gradient of w is one element that sums df over everything, nk times."""
    b = Builder("all_terms", [ni, nj], 1, ["w", "y"], [[1], [ni, nj, nk]])
    y = b.load("y", [[1, 0, 0], [0, 1, 0], [0, 0, 1]])
    b.sum(2, 0, nk - 1, b.bin("add", b.load("w", [[0, 0, 0]]), y))
    return b.done()


def test_products_are_reordered():
    assert "; factored" in Plan(_product(600, 40, 300)).disassemble(-1)
    # no auxiliary kernel sums a whole tensor on its own
    e = _all_terms(500, 600, 20)
    plan = Plan(e)
    w = next(q for q, a in enumerate(e.accesses) if a.arg == 0)
    assert "; auxiliary kernel" not in plan.disassemble(w)


@pytest.mark.gpu
@pytest.mark.parametrize("make", [lambda: _product(600, 40, 300), lambda: _all_terms(500, 600, 20)])
def test_reordered_products(make):
    from tests.gpu_util import check_against_oracle
    e = make()
    args, df = W.make_inputs(e, ("uniform", -0.5, 0.5), seed=3)
    check_against_oracle(e, args, df, nthreads=max_threads())
