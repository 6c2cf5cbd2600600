"""Tile programs (sums of a term that couples two variables, as written) against the oracle: edges of tiles in every direction,
groups of threads and blocks that share a sum, summed columns, further output variables, operands that are expressions, a core that is
read step by step (all of its steps: test_gpu_tile_cores.py), strides and reversed reads, inputs that are not 16-byte aligned."""
import pytest
import torch

from oracle.oracle import Oracle, max_threads
from paper_1711_01348_b200 import Plan
from workloads import configs as W
from workloads.expr import Builder, unit


def _functions(ni, nj, nk):
    """f_ij = exp(0.1 s), s = sum_k tanh(x_ik y_jk + w_i) (y_jk - x_ik) / (1.5 + v_k^2)"""
    b = Builder("functions", [ni, nj], 1, ["x", "y", "w", "v"], [[ni, nk], [nj, nk], [ni], [nk]])
    x, y = b.load("x", [unit(3, (0, 1)), unit(3, (2, 1))]), b.load("y", [unit(3, (1, 1)), unit(3, (2, 1))])
    w, v = b.load("w", [unit(3, (0, 1))]), b.load("v", [unit(3, (2, 1))])
    t = b.bin("mul", b.un("tanh", b.bin("add", b.bin("mul", x, y), w)), b.bin("sub", y, x))
    t = b.bin("mul", t, b.bin("div", b.const(1.0), b.bin("add", b.powi(v, 2), b.const(1.5))))
    b.un("exp", b.bin("mul", b.sum(2, 0, nk - 1, t), b.const(0.1)))
    return b.done()


def _planes(nm, ni, nj, nk):
    """f_mij = sum_k (x_mik - y_{j, nk-1-k})^2 w_m + 0.5 z_{2k} x_mik: a third output variable, a reversed and a strided read"""
    b = Builder("planes", [nm, ni, nj], 1, ["x", "y", "w", "z"], [[nm, ni, nk], [nj, nk], [nm], [2 * nk]])
    x = b.load("x", [unit(4, (0, 1)), unit(4, (1, 1)), unit(4, (3, 1))])
    y = b.load("y", [unit(4, (2, 1)), unit(4, (3, -1))], [0, nk - 1])
    w, z = b.load("w", [unit(4, (0, 1))]), b.load("z", [unit(4, (3, 2))])
    b.sum(3, 0, nk - 1, b.bin("add", b.bin("mul", b.powi(b.bin("sub", x, y), 2), w), b.bin("mul", b.bin("mul", z, x), b.const(0.5))))
    return b.done()


CASES = {
    "ragged": lambda: W.intro(257, 129, 13),
    "one_over": lambda: W.intro(1025, 65, 7),
    "shortest_sum": lambda: W.intro(97, 1031, 4),
    "few_rows": lambda: W.intro(5, 9001, 9),
    "few_columns": lambda: W.intro(9001, 5, 9),
    "long_pieces": lambda: W.intro(33, 31, 1201),
    "aligned": lambda: W.intro(512, 256, 16),
    "two_to_the_24": lambda: W.intro(1024, 512, 32),
    "short_and_large": lambda: W.intro(4500, 2700, 5),
    "functions": lambda: _functions(411, 253, 9),
    "planes": lambda: _planes(3, 290, 77, 11),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_taken(name):
    e = CASES[name]()
    plan = Plan(e)
    text = "".join(plan.disassemble(w) for w in [-1] + [-2 - s for s in range(plan.num_stages())] + list(range(len(e.accesses))))
    assert text.count("; tile program") >= (1 if name in ("functions", "planes") else 2 if name == "short_and_large" else 3)


@pytest.mark.gpu
@pytest.mark.parametrize("name", sorted(CASES))
def test_tile_programs(name):
    from tests.gpu_util import check_against_oracle
    e = CASES[name]()
    # (sums of 1201 terms of up to 0.5 leave the range of exp; of up to 0.2^2 0.1 + 0.1^3 they stay below 7)
    r = 0.1 if name == "long_pieces" else 0.5
    args, df = W.make_inputs(e, ("uniform", -r, r), seed=5)
    check_against_oracle(e, args, df, nthreads=max_threads())


@pytest.mark.gpu
def test_inputs_off_by_four_bytes():
    from tests.gpu_util import assert_close
    e = W.intro(512, 256, 16)
    args, df = W.make_inputs(e, ("uniform", -0.5, 0.5), seed=6)
    shift = lambda t: torch.cat([torch.zeros(1), t.flatten()]).cuda()[1:]
    a, d = [shift(t) for t in args], shift(df)
    f, g = shift(torch.full(e.out_shape, float("nan"))), [shift(torch.full(s, float("nan"))) for s in e.arg_shapes]
    plan = Plan(e)
    ws = torch.zeros(max(256, plan.workspace_bytes()), dtype=torch.uint8, device="cuda")
    plan.forward([t.data_ptr() for t in a], f.data_ptr(), 0, ws.data_ptr(), ws.numel())
    plan.backward([t.data_ptr() for t in a], d.data_ptr(), [t.data_ptr() for t in g], ws.data_ptr(), ws.numel())
    torch.cuda.synchronize()
    orc = Oracle(e)
    want, scale = orc.forward(args, nthreads=max_threads())
    assert_close(f.cpu().numpy().reshape(e.out_shape), want, scale, "f")
    dx, terms = orc.backward(args, df, nthreads=max_threads())
    for t, w, s in zip(g, dx, terms):
        assert_close(t.cpu().numpy().reshape(w.shape), w, s, "gradient")
