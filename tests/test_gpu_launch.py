"""Launch order: overlapped starts of consecutive kernels, captured graphs and concurrent streams give the same bits."""
import pytest
import torch

from workloads import configs as W

pytestmark = pytest.mark.gpu

from tests.gpu_util import GpuRun  # noqa: E402


def _step(run, stream):
    ptrs = [a.data_ptr() for a in run.args]
    run.plan.forward(ptrs, run.f.data_ptr(), stream, run.ws.data_ptr(), run.ws.numel())
    run.plan.backward(ptrs, run.df.data_ptr(), [d.data_ptr() for d in run.dargs], run.ws.data_ptr(), run.ws.numel(), stream)


@pytest.mark.parametrize("make", [lambda: W.intro(64, 64, 5), lambda: W.intro(700, 900, 33), lambda: W.shifted(301)])
def test_captured_and_concurrent_steps(make):
    e = make()
    runs = [GpuRun(e, *W.make_inputs(e, ("uniform", -0.5, 0.5), seed=s)) for s in (1, 2)]
    want = []
    for r in runs:
        _step(r, torch.cuda.current_stream().cuda_stream)
        torch.cuda.synchronize()
        want.append([t.clone() for t in [r.f] + r.dargs])
    streams = [torch.cuda.Stream() for _ in runs]
    for _ in range(10):
        for r, s in zip(runs, streams):
            _step(r, s.cuda_stream)
    torch.cuda.synchronize()
    for r, w in zip(runs, want):
        assert all(torch.equal(a, b) for a, b in zip([r.f] + r.dargs, w))
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        _step(runs[0], torch.cuda.current_stream().cuda_stream)
    for t in [runs[0].f] + runs[0].dargs:
        t.fill_(float("nan"))
    graph.replay()
    torch.cuda.synchronize()
    assert all(torch.equal(a, b) for a, b in zip([runs[0].f] + runs[0].dargs, want[0]))


def test_shared_auxiliaries_follow_the_call():
    """Row sums and contractions that several gradients need are computed once per backward call, and again by every call:
    new df, new arguments, subsets and single gradients never see the values of an earlier call."""
    e = W.intro(600, 700, 60)
    runs = [GpuRun(e, *W.make_inputs(e, ("uniform", -0.5, 0.5), seed=s)) for s in (1, 2)]
    want = [r.backward() for r in runs]
    a = runs[0]
    st = torch.cuda.current_stream().cuda_stream
    for other in (1, 0):
        ptrs = [t.data_ptr() for t in runs[other].args]
        df = runs[other].df.data_ptr()
        a.plan.backward_stage(ptrs, df, a.ws.data_ptr(), a.ws.numel(), st)
        for p in (3, 2, 0, 1):
            a.plan.backward_arg(ptrs, df, p, a.dargs[p].data_ptr(), a.ws.data_ptr(), a.ws.numel(), st)
        torch.cuda.synchronize()
        for d, w in zip(a.dargs, want[other]):
            assert torch.equal(d.cpu(), torch.from_numpy(w))
        for wanted in ([False, False, True, True], [True, False, True, False]):
            a.plan.backward(ptrs, df, [d.data_ptr() if k else 0 for d, k in zip(a.dargs, wanted)], a.ws.data_ptr(), a.ws.numel(), st)
            torch.cuda.synchronize()
            for d, w in zip(a.dargs, want[other]):
                assert torch.equal(d.cpu(), torch.from_numpy(w))
