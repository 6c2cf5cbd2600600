"""Contractions whose summation is split need room for planes of partial sums, but can run in fewer shares: a forward pass without
a workspace and a backward pass on the built-in scratch are accepted as they were before any contraction was split."""
import pytest
import torch

from paper_1711_01348_b200 import Plan, TadError
from workloads import configs as W

# (forward passes that are split; 708 x 6661 outputs of 5186 terms, whose planes are larger than the built-in scratch)
FORWARD = [lambda: W.ex_matmul(176, 550, 41), lambda: W.conv1d(2, 210, 7, 878, 5), lambda: W.ex_matmul(300, 5000, 200)]
BUILT_IN = [lambda: W.ex_matmul(708, 6661, 5186), lambda: W.ex_matmul(130, 9000, 140), lambda: W.intro(900, 1000, 21)]


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
