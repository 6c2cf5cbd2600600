"""Line sums whose lanes walk in step: ranges that move with the lane, lane strides and skews, one and two loops, rows
shorter than a warp, shares that take several pieces, squared loads and one to four loads per term."""
import pytest

from oracle.oracle import max_threads
from workloads import configs as W
from workloads.expr import Builder

pytestmark = pytest.mark.gpu

from tests.gpu_util import GpuRun, check_against_oracle  # noqa: E402


def _strided(n, m, a, c, extra):
    """f_ij = x_{a i + c j} w_j^2 (v_i): the gradient of x sums df over the lattice a i + c j = beta."""
    b = Builder(f"lattice_{a}_{c}", [n, m], 0, ["x", "w", "v"], [[a * (n - 1) + c * (m - 1) + 1], [m], [n]])
    p = b.bin("mul", b.load("x", [[a, c]]), b.powi(b.load("w", [[0, 1]]), 2))
    b.bin("mul", p, b.load("v", [[1, 0]])) if extra else None
    return b.done()


def _few_elements(n, nj, nk):
    """f_i = sum_jk x_{j+k} y_{i+j} with x as long as the output: nj + nk - 1 elements of its gradient have terms."""
    b = Builder("few_elements", [n], 2, ["x", "y"], [[n], [n + nj]])
    p = b.bin("mul", b.load("x", [[0, 1, 1]]), b.load("y", [[1, 1, 0]]))
    b.sum(1, 0, nj - 1, b.sum(2, 0, nk - 1, p))
    return b.done()


def _short_runs(n, m, k):
    """f_ij = sum_k x_{i+k} w_{j+k}: the gradient of x walks m runs of at most k terms."""
    b = Builder("short_runs", [n, m], 1, ["x", "w"], [[n + k - 1], [m + k - 1]])
    b.sum(2, 0, k - 1, b.bin("mul", b.load("x", [[1, 0, 1]]), b.load("w", [[0, 1, 1]])))
    return b.done()


CASES = {
    "bounds_move_with_the_lane": lambda: W.shifted(777),
    "short_rows": lambda: W.nonunimodular(21),
    "two_loops": lambda: W.nonunimodular(83),
    "stride_2": lambda: _strided(700, 501, 2, 3, True),
    "stride_5": lambda: _strided(400, 611, 3, 5, True),
    "negative_direction": lambda: _strided(601, 350, 5, 2, False),
    "no_unit_lanes": lambda: _strided(90, 80, 11, 13, True),
    "one_lane_wide": lambda: _strided(1500, 1, 1, 1, True),
    "many_pieces": lambda: _strided(9, 40000, 1, 1, True),
    "few_elements": lambda: _few_elements(30001, 6, 29),
    "short_runs": lambda: _short_runs(1500, 90, 3),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_line_sums(name):
    e = CASES[name]()
    args, df = W.make_inputs(e, ("uniform", -1, 1), seed=5)
    run = GpuRun(e, args, df)
    assert any("; line sums" in run.plan.disassemble(w) for w in range(len(e.accesses)))
    check_against_oracle(e, args, df, nthreads=max_threads())
