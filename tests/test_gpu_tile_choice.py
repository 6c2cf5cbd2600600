"""Sums that couple two variables: where tiles run them, and where point programs, contractions or the interpreter do."""
import pytest

from oracle.oracle import max_threads
from paper_1711_01348_b200 import Plan
from workloads import configs as W
from workloads.expr import Builder, unit


def _pair(term, ni, nj, nk, nz=0):
    """f_[z]ij = sum_k term(x_[z]ik, y_[z]jk)"""
    o = 1 if nz else 0
    n, z, zr = 3 + o, [nz] * o, [unit(3 + o, (0, 1))] * o
    b = Builder("pair", z + [ni, nj], 1, ["x", "y"], [z + [ni, nk], z + [nj, nk]])
    x = b.load("x", zr + [unit(n, (o, 1)), unit(n, (o + 2, 1))])
    b.sum(o + 2, 0, nk - 1, term(b, x, b.load("y", zr + [unit(n, (o + 1, 1)), unit(n, (o + 2, 1))])))
    return b.done()


def _two_products(ni, nj, nk):
    """f_ij = sum_k x_ik y_jk + u_ik v_jk"""
    b = Builder("products", [ni, nj], 1, ["x", "y", "u", "v"], [[ni, nk], [nj, nk]] * 2)
    x, y, u, v = (b.load(n, [unit(3, (i % 2, 1)), unit(3, (2, 1))]) for i, n in enumerate("xyuv"))
    b.sum(2, 0, nk - 1, b.bin("add", b.bin("mul", x, y), b.bin("mul", u, v)))
    return b.done()


def _square(b, x, y):
    return b.powi(b.bin("add", x, y), 2)


def _sum(b, x, y):
    return b.bin("add", x, y)


def _tanh(b, x, y):
    return b.un("tanh", b.bin("mul", x, y))


# expression, what runs the forward pass, what runs the gradients
CASES = {
    "products": (lambda: _two_products(340, 340, 340), "contraction", "contraction"),
    "products_line": (lambda: _two_products(256, 256, 256), "tile program", None),
    "products_past_it": (lambda: _two_products(256, 256, 257), "contraction", None),
    "exact_parts": (lambda: _pair(_sum, 700, 400, 16), "tile program", None),
    "squares": (lambda: _pair(_square, 300, 300, 300), "tile program", "tile program"),
    "small_squares": (lambda: _pair(_square, 64, 64, 17), "tile program", "tile program"),
    "batches_of_squares": (lambda: _pair(_square, 4, 4, 8, 2000), "point program", "point program"),
    "batches_of_tanh": (lambda: _pair(_tanh, 4, 4, 8, 2000), "point program", "point program"),
    "odd_batches": (lambda: _pair(_tanh, 3, 5, 7, 3000), "point program", "point program"),
    "large_batches": (lambda: _pair(_tanh, 16, 16, 16, 200), "tile program", "tile program"),
    "small_tanh": (lambda: _pair(_tanh, 64, 64, 17), "tile program", "point program"),
    "wide_tanh": (lambda: _pair(_tanh, 64, 1000, 17), "tile program", "tile program"),
    "many_short_sums": (lambda: _pair(_sum, 5, 3655, 4, 149), "vars=", None),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_taken(name):
    build, forward, gradients = CASES[name]
    e = build()
    plan = Plan(e)
    assert forward in plan.disassemble(-1)
    assert (forward == "tile program") == ("tile program" in plan.disassemble(-1))
    for q in range(len(e.accesses)) if gradients else []:
        assert gradients in plan.disassemble(q), q


@pytest.mark.gpu
@pytest.mark.parametrize("name", sorted(CASES))
def test_choice(name):
    from tests.gpu_util import check_against_oracle
    e = CASES[name][0]()
    check_against_oracle(e, *W.make_inputs(e, ("uniform", -0.9, 0.9), seed=4), nthreads=max_threads())
