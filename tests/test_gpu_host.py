"""tad_step_host where an argument is read along one line only (a diagonal, a strided vector): single elements travel, the
rest of the gradient is zero whatever the buffer held; tensors read in full and lines with offsets and sums beside them."""
import numpy as np
import pytest
import torch

from oracle.oracle import Oracle, max_threads
from workloads import configs as W
from workloads.expr import Builder

pytestmark = pytest.mark.gpu

from paper_1711_01348_b200 import Plan  # noqa: E402
from tests.gpu_util import assert_close  # noqa: E402


def _lines(n, k):
    """f_i = sum_k x_{70 i + 3} y_{i+1, n-i} z_k: a strided vector with an offset, an antidiagonal, a tensor read in full."""
    b = Builder("lines", [n], 1, ["x", "y", "z"], [[70 * n + 9], [n + 2, n + 1], [k]])
    p = b.bin("mul", b.load("x", [[70, 0]], [3]), b.load("y", [[1, 0], [-1, 0]], [1, n]))
    b.sum(1, 0, k - 1, b.bin("mul", p, b.load("z", [[0, 1]])))
    return b.done()


@pytest.mark.parametrize("saved", [False, True])
@pytest.mark.parametrize("make", [lambda: W.intro(131, 97, 5), lambda: W.intro(201, 97, 5), lambda: _lines(200, 7), lambda: W.ex_matmul(65, 70, 33)])
def test_step_host(make, saved):
    e = make()
    args, df = W.make_inputs(e, ("uniform", -0.5, 0.5), seed=4)
    plan = Plan(e, saved_forward=saved)
    pin = [t.pin_memory() for t in args + [df]]
    f = torch.full(list(e.out_shape), 7.0).pin_memory()
    dargs = [torch.full(list(s), 7.0).pin_memory() for s in e.arg_shapes]
    ws = torch.full((plan.staging_bytes(),), 255, dtype=torch.uint8, device="cuda")      # every float of it a NaN
    for _ in range(2):
        plan.step_host([t.data_ptr() for t in pin[:-1]], pin[-1].data_ptr(), f.data_ptr(), [d.data_ptr() for d in dargs],
                       ws.data_ptr(), ws.numel(), torch.cuda.current_stream().cuda_stream)
    orc = Oracle(e)
    f_o, fabs = orc.forward(args, nthreads=max_threads())
    dx_o, t_o = orc.backward(args, df, nthreads=max_threads())
    assert_close(f.numpy(), f_o, fabs, "f")
    for d, o, t, n in zip(dargs, dx_o, t_o, e.arg_names):
        assert_close(d.numpy(), o, t, "d" + n)
        assert np.all(d.numpy()[t == 0] == 0.0)
