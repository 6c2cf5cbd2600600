"""Contractions whose summation is split need room for planes of partial sums, but can run in fewer shares: a forward pass without
a workspace and a backward pass on the built-in scratch are accepted as they were before any contraction was split.  So are sums
that are pushed inside or split where a kernel of their own, which needs no room, is slower."""
import pytest
import torch

from paper_1711_01348_b200 import Plan, TadError
from workloads import configs as W
from workloads.expr import Builder, unit


def _two_products(ni, nj, nk, weighted=False):
    """f_ij = [w_ij] sum_k x_ik y_jk + u_ik v_jk"""
    b = Builder("products", [ni, nj], 1, ["x", "y", "u", "v", "w"][:5 if weighted else 4], [[ni, nk], [nj, nk], [ni, nk], [nj, nk], [ni, nj]][:5 if weighted else 4])
    x, y, u, v = (b.load(n, [unit(3, (i % 2, 1)), unit(3, (2, 1))]) for i, n in enumerate("xyuv"))
    s = b.sum(2, 0, nk - 1, b.bin("add", b.bin("mul", x, y), b.bin("mul", u, v)))
    if weighted:
        b.bin("mul", b.load("w", [unit(3, (0, 1)), unit(3, (1, 1))]), s)
    return b.done()


def _rows(n, k):
    """f_i = sum_k y_ik w_k"""
    b = Builder("rows", [n], 1, ["y", "w"], [[n, k], [k]])
    b.sum(1, 0, k - 1, b.bin("mul", b.load("y", [unit(2, (0, 1)), unit(2, (1, 1))]), b.load("w", [unit(2, (1, 1))])))
    return b.done()


# (forward passes that are split; 708 x 6661 outputs of 5186 terms, whose planes are larger than the built-in scratch)
FORWARD = [lambda: W.ex_matmul(176, 550, 41), lambda: W.conv1d(2, 210, 7, 878, 5), lambda: W.ex_matmul(300, 5000, 200)]
# (sums of products pushed inside, long rows split: as tiles and a block a row they need no tensors and planes)
FORWARD += [lambda: _two_products(340, 340, 340), lambda: _two_products(1000, 700, 40, True), lambda: _rows(36, 300000)]
BUILT_IN = [lambda: W.ex_matmul(708, 6661, 5186), lambda: W.ex_matmul(130, 9000, 140), lambda: W.intro(900, 1000, 21)]
BUILT_IN += [lambda: _two_products(2000, 2000, 12), lambda: _two_products(2000, 2000, 12, True)]


@pytest.mark.skipif(torch.cuda.is_available(), reason="fake pointers must not reach a GPU")
@pytest.mark.parametrize("make", FORWARD)
def test_forward_without_workspace_is_accepted(make):
    e = make()
    with pytest.raises(TadError) as ei:
        Plan(e).forward([1 << 20] * len(e.arg_shapes), 1 << 20)
    assert ei.value.code == "TAD_ERR_CUDA"                      # past the checks, and there is no device


@pytest.mark.skipif(torch.cuda.is_available(), reason="fake pointers must not reach a GPU")
@pytest.mark.parametrize("make", BUILT_IN)
def test_built_in_scratch_is_accepted(make):
    e = make()
    with pytest.raises(TadError) as ei:
        Plan(e).backward_noalloc([1 << 20] * len(e.arg_shapes), 1 << 20, [1 << 20] * len(e.arg_shapes))
    assert ei.value.code == "TAD_ERR_CUDA"


@pytest.mark.gpu
@pytest.mark.parametrize("make", FORWARD)
def test_forward_without_workspace(make):
    from tests.gpu_util import GpuRun
    e = make()
    run = GpuRun(e, *W.make_inputs(e, ("normal", 0, 1), seed=2))
    want = run.forward()
    run.f.fill_(float("nan"))
    run.plan.forward([a.data_ptr() for a in run.args], run.f.data_ptr(), torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    assert float(abs(run.f.cpu().numpy() - want).max()) <= 1e-5 * float(abs(want).max())


@pytest.mark.gpu
@pytest.mark.parametrize("make", BUILT_IN)
def test_built_in_scratch(make):
    from tests.gpu_util import GpuRun
    e = make()
    run = GpuRun(e, *W.make_inputs(e, ("uniform", -0.5, 0.5), seed=2))
    want = run.backward()
    for d in run.dargs:
        d.fill_(float("nan"))
    run.plan.backward_noalloc([a.data_ptr() for a in run.args], run.df.data_ptr(), [d.data_ptr() for d in run.dargs],
                              torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    for d, w in zip(run.dargs, want):
        assert float(abs(d.cpu().numpy() - w).max()) <= 1e-5 * float(abs(w).max())
