"""Products of loads: rows that follow one another (one long row, in runs along it, with every remainder), rows that do not, reads
along and against the row, single reads a row, strides, powers, wide and narrow pieces, tensors off a 16-byte boundary."""
import pytest
import torch

from oracle.oracle import Oracle, max_threads
from paper_1711_01348_b200 import Plan
from workloads import configs as W
from workloads.expr import Builder, unit


def _flat(ni, nj):
    """f_ij = x_ij y_ij^2: one row of ni nj"""
    b = Builder("flat", [ni, nj], 0, ["x", "y"], [[ni, nj], [ni, nj]])
    x, y = [b.load(n, [unit(2, (0, 1)), unit(2, (1, 1))]) for n in "xy"]
    b.bin("mul", x, b.powi(y, 2))
    return b.done()


def _rows(ni, nj, pad):
    """f_ij = x_ij y_{nj-1-j} w_i (v_{i, 2j}): a padded operand, a reversed, a single and a strided read"""
    b = Builder("rows", [ni, nj], 0, ["x", "y", "w", "v"], [[ni, nj + pad], [nj], [ni], [ni, 2 * nj]])
    x = b.load("x", [unit(2, (0, 1)), unit(2, (1, 1))])
    y = b.load("y", [unit(2, (1, -1))], [nj - 1])
    w = b.load("w", [unit(2, (0, 1))])
    v = b.load("v", [unit(2, (0, 1)), unit(2, (1, 2))])
    b.bin("mul", b.bin("mul", x, y), b.bin("mul", b.powi(w, 3), v) if pad % 2 else w)
    return b.done()


def _cube(n, m):
    """f_ijk = x_{2i+j, j-k+m-1} y_{i, j, k}: rows of a table against the run, an operand of the output's shape"""
    b = Builder("cube", [n, n, m], 0, ["x", "y"], [[3 * n - 2, n + m - 1], [n, n, m]])
    x = b.load("x", [unit(3, (0, 2), (1, 1)), unit(3, (1, 1), (2, -1))], [0, m - 1])
    b.bin("mul", x, b.load("y", [unit(3, (0, 1)), unit(3, (1, 1)), unit(3, (2, 1))]))
    return b.done()


def _line(n, off, loads):
    """f_i = x_i y_{n-1-i} w_{i+off}, the first `loads` of them: one row, a piece or several a thread"""
    b = Builder("line", [n], 0, ["x", "y", "w"][:loads], [[n], [n], [n + off]][:loads])
    r = b.load("x", [unit(1, (0, 1))])
    if loads > 1:
        r = b.bin("mul", r, b.load("y", [unit(1, (0, -1))], [n - 1]))
    b.bin("mul", r, b.load("w", [unit(1, (0, 1))], [off])) if loads > 2 else b.bin("mul", r, b.const(2.0))
    return b.done()


CASES = {
    "flat_1": lambda: _flat(3, 1), "flat_7": lambda: _flat(1, 7), "flat_small": lambda: _flat(33, 31), "flat_odd": lambda: _flat(1301, 2477),
    "flat_run": lambda: _flat(2048, 2049), "flat_remainder": lambda: _flat(1025, 4099), "flat_aligned": lambda: _flat(1024, 4096),
    "rows_aligned": lambda: _rows(900, 1024, 0), "rows_padded": lambda: _rows(911, 1024, 4), "rows_odd": lambda: _rows(901, 1023, 1),
    "rows_short": lambda: _rows(4099, 5, 3), "cube_aligned": lambda: _cube(96, 128), "cube_even": lambda: _cube(90, 130), "cube_odd": lambda: _cube(97, 129),
}


def _check(e, shift=0):
    from tests.gpu_util import assert_close
    args, df = W.make_inputs(e, ("normal", 0, 1), seed=3)
    dev = lambda t: torch.cat([torch.zeros(shift), t.flatten()]).cuda()[shift:]
    a, d = [dev(t) for t in args], dev(df)
    f, g = dev(torch.full(e.out_shape, float("nan"))), [dev(torch.full(s, float("nan"))) for s in e.arg_shapes]
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


@pytest.mark.gpu
@pytest.mark.parametrize("name", sorted(CASES))
def test_products(name):
    _check(CASES[name]())


@pytest.mark.gpu
@pytest.mark.parametrize("loads", [1, 2, 3])
@pytest.mark.parametrize("n,off", [(3, 1), (1024, 4), (1027, 2), (100001, 1), (600000, 4), (2424831, 2), (2424836, 4)])
def test_one_row(n, off, loads):
    _check(_line(n, off, loads))


@pytest.mark.gpu
@pytest.mark.parametrize("name", ["flat_run", "rows_aligned", "cube_aligned"])
@pytest.mark.parametrize("shift", [1, 2])
def test_off_a_boundary(name, shift):
    _check(CASES[name](), shift)


@pytest.mark.gpu
@pytest.mark.parametrize("ni,nj", [(70, 5001), (600, 1000), (1000, 4003)])
def test_repeated(ni, nj):
    """the gradient of x in f_i = sum_j w_i x_ij repeats w_i df_i (w inside the sum: f, which nearly cancels, is then measured by its
    terms; of 4003 of them it is off by some 4003^(1/2) 2^-24 60, 1.4e-5 where |f| may be 0.02)"""
    b = Builder("repeated", [ni], 1, ["x", "w"], [[ni, nj], [ni]])
    b.sum(1, 0, nj - 1, b.bin("mul", b.load("w", [unit(2, (0, 1))]), b.load("x", [unit(2, (0, 1)), unit(2, (1, 1))])))
    e = b.done()
    assert "element-wise" in Plan(e).disassemble(0) or "element-wise" in Plan(e).disassemble(1)
    _check(e)


def test_rows_are_joined():
    assert "rows of %d along" % (1301 * 2477) in Plan(_flat(1301, 2477)).disassemble(-1)
