"""Row sums, plain and weighted, by a warp and by a block a row: rows that start off a 16-byte boundary, weights that start off
another one than the rows, lengths around the pieces of a warp and of a block, strided weights, the first sizes of either rule."""
import pytest

from oracle.oracle import max_threads
from paper_1711_01348_b200 import Plan
from workloads import configs as W
from workloads.expr import Builder, unit

CASES = [(32, 512, 1), (33, 513, 1), (150, 2823, 1), (264, 4099, 2), (1183, 515, 1), (1185, 514, 1), (1024, 7, 1), (1030, 4097, 1), (2000, 1031, 3)]


def _weighted(n, k, step):
    """f_i = sum_k y_ik w_{step k + 1}"""
    b = Builder("weighted", [n], 1, ["y", "w"], [[n, k], [step * k + 1]])
    b.sum(1, 0, k - 1, b.bin("mul", b.load("y", [unit(2, (0, 1)), unit(2, (1, 1))]), b.load("w", [unit(2, (1, step))], [1])))
    return b.done()


# an element a lane or pieces, a warp or a block a row: either side of each line
EDGES = [(2001, 32, 1), (2001, 33, 1), (1500, 32, 2), (1500, 33, 2), (1200, 65, 1), (250, 999, 1), (250, 1000, 1), (1183, 4731, 1), (1183, 4732, 1), (1184, 4736, 1), (296, 1185, 1), (297, 1189, 1), (2368, 601, 1), (2369, 601, 1)]


@pytest.mark.parametrize("n,k,step", CASES)
def test_taken(n, k, step):
    assert "row sums" in Plan(_weighted(n, k, step)).disassemble(-1)


# fewer rows than SMs, too long for a block each: (30000 + 800 n) elements are the last
@pytest.mark.parametrize("n,k,rows", [(40, 62000, True), (40, 62001, False), (147, 147600, True), (147, 147601, False), (148, 200000, True), (32, 1000000, False)])
def test_long_rows_are_split(n, k, rows):
    assert ("row sums" in Plan(_weighted(n, k, 1)).disassemble(-1)) == rows


@pytest.mark.gpu
@pytest.mark.parametrize("n,k,step", CASES + EDGES + [(40, 62000, 1), (40, 62001, 1)])
def test_weighted_rows(n, k, step):
    from tests.gpu_util import check_against_oracle
    e = _weighted(n, k, step)
    check_against_oracle(e, *W.make_inputs(e, ("normal", 0, 1), seed=k), nthreads=max_threads())


@pytest.mark.gpu
@pytest.mark.parametrize("n,nj,nk", [(70, 2001, 40), (1300, 517, 8)])
def test_plain_rows(n, nj, nk):
    """the gradient of d in the intro expression sums rows of the staged adjoint"""
    from tests.gpu_util import check_against_oracle
    e = W.intro(n, nj, nk)
    assert "row sums" in Plan(e).disassemble(3)
    check_against_oracle(e, *W.make_inputs(e, ("uniform", -0.5, 0.5), seed=n), nthreads=max_threads())
