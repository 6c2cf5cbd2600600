"""Rounding of long line sums: the terms of a piece are added up in four chains of sixteen, whole pieces behind them.  Terms that
are all alike show the longest chain, since its additions round the same way: 16 additions and 2 for the four chains of a piece,
each off by at most 2^-24 of its result, and a few for the sums of pieces, which differ in size.  Chains through all pieces of
a share are off by three times as much."""
import pytest
import torch

from workloads.expr import Builder

pytestmark = pytest.mark.gpu

from tests.gpu_util import GpuRun  # noqa: E402


@pytest.mark.parametrize("n,m,k", [(4096, 4096, 1), (512, 512, 512), (256, 256, 256)])
def test_sums_of_like_terms(n, m, k):
    """f_ijl = x_i+j y_l: the gradient of x sums n m k terms of about 1 / 3 along the lattice, that of y all of them."""
    b = Builder("like_terms", [n, m, k] if k > 1 else [n, m], 0, ["x", "y"], [[n + m - 1], [k]])
    pad = [0] if k > 1 else []
    b.bin("mul", b.load("x", [[1, 1] + pad]), b.load("y", [[0, 0] + ([1] if k > 1 else [])]))
    e = b.done()
    third = torch.tensor(1 / 3)
    args = [torch.full((n + m - 1,), 1.0), torch.full((k,), 1.0)]
    df = third.expand(e.out_shape).contiguous()
    dx, dy = GpuRun(e, args, df).backward()
    i = torch.arange(n + m - 1)
    terms = torch.minimum(torch.minimum(i + 1, n + m - 1 - i), torch.tensor(min(n, m))).double() * k
    for got, count in ((dx, terms), (dy, torch.full((k,), float(n * m)))):
        want = count * third.double()
        rel = ((torch.from_numpy(got).double() - want).abs() / want).max()
        assert float(rel) <= 20 * 2.0 ** -24, float(rel) * 2 ** 24
