"""Point programs (general terms over small index spaces) against the oracle: one and four points per thread, single and
many term lanes, ragged last batches, shares of the terms, deep stacks and temporaries, empty prefixes, scalar outputs."""
import pytest

from oracle.oracle import max_threads
from workloads import configs as W
from workloads.expr import Builder, unit

pytestmark = pytest.mark.gpu

from tests.gpu_util import GpuRun, check_against_oracle  # noqa: E402


def _shared_sum(ni, nj, nk):
    """f_ij = tanh(s) (w_i + s), s = sum_k (sin(x_i y_jk) + x_i): a value of a sum used twice, gradients over i, over (j, k)."""
    b = Builder("shared_sum", [ni, nj], 1, ["x", "y", "w"], [[ni], [nj, nk], [ni]])
    x = b.load("x", [unit(3, (0, 1))])
    w = b.load("w", [unit(3, (0, 1))])
    y = b.load("y", [unit(3, (1, 1)), unit(3, (2, 1))])
    s = b.sum(2, 0, nk - 1, b.bin("add", b.un("sin", b.bin("mul", x, y)), x))
    b.bin("mul", b.un("tanh", s), b.bin("add", w, s))
    return b.done()


CASES = {
    "one_output": lambda: W.intro(1, 1, 1),
    "one_term": lambda: W.intro(9, 1, 1),
    "odd_batches": lambda: W.intro(33, 131, 3),
    "lanes_64": lambda: W.intro(64, 64, 5),
    "few_outputs_many_terms": lambda: W.intro(2, 3001, 2),
    "many_outputs": lambda: W.intro(1999, 67, 3),
    "shares": lambda: W.ex_all_ops(60001),
    "four_points": lambda: W.ex_all_ops(131073),
    "shared_sum": lambda: _shared_sum(37, 53, 6),
    # the sum as terms and a tail behind it: values before, inside and behind the sum, at few and at many outputs
    "tail_behind_sum": lambda: _shared_sum(3, 7, 45),
    "tail_many_outputs": lambda: _shared_sum(151, 400, 4),
    "tail_all_functions": lambda: W.intro(40, 31, 33),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_point_programs(name):
    e = CASES[name]()
    args, df = W.make_inputs(e, ("uniform", -0.5, 0.5), seed=11)
    run = GpuRun(e, args, df)
    parts = [-1] + [-2 - s for s in range(run.plan.num_stages())] + list(range(len(e.accesses)))
    assert any("; point program" in run.plan.disassemble(w) for w in parts)
    check_against_oracle(e, args, df, nthreads=max_threads())
