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
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_line_sums(name):
    e = CASES[name]()
    args, df = W.make_inputs(e, ("uniform", -1, 1), seed=5)
    run = GpuRun(e, args, df)
    assert any("; line sums" in run.plan.disassemble(w) for w in range(len(e.accesses)))
    check_against_oracle(e, args, df, nthreads=max_threads())
