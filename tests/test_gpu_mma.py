"""Tensor-core contraction kernel: tile edges, every gather mode, splits, guards, non-finite operands.

Tolerance per output, relative to the sum of |terms|: the products left out by the three-way bf16 split 2^-23, four
truncated accumulator steps per stage of 64 summation indices (each below 2^-23 of a partial sum, the steps of the small
products below one more together), one rounding 2^-24 per stage for the running sum and per plane: (8 + stages) 2^-23
bounds them all."""
import math

import pytest
import torch

from paper_1711_01348_b200 import Plan
from workloads import configs as W

pytestmark = pytest.mark.gpu

from tests.gpu_util import GpuRun  # noqa: E402


def _close(got, want, scale, n_terms, what):
    tol = (8 + math.ceil(n_terms / 64)) * 2.0 ** -23 * scale + 1e-45
    err = (torch.from_numpy(got).double() - want).abs()
    assert bool((err <= tol).all()), f"{what}: worst {float((err / tol).max()):.2f} of the tolerance"


# (rows, summed, columns): tile and stage edges, remainders of the 16-wide steps, a split summation, wide and narrow sides
SIZES = [(128, 64, 128), (127, 63, 129), (129, 65, 127), (257, 17, 64), (64, 130, 257), (8, 2050, 300), (300, 333, 65),
         (513, 16, 700), (160, 5000, 136)]


@pytest.mark.parametrize("transposed", [False, True])
@pytest.mark.parametrize("ni,nk,nj", SIZES)
def test_matrix_products(ni, nk, nj, transposed):
    e = W.ex_matmul_t(ni, nj, nk) if transposed else W.ex_matmul(ni, nk, nj)
    args, df = W.make_inputs(e, ("normal", 0, 1), seed=ni + nk)
    run = GpuRun(e, args, df)
    f = run.forward()
    dx, dy = run.backward()
    x, y, d = args[0].double(), args[1].double(), df.double()
    y = y.T if transposed else y                                # summed x columns
    _close(f, x @ y, x.abs() @ y.abs(), nk, "forward")
    _close(dx, d @ y.T, d.abs() @ y.T.abs(), nj, "dx")
    want, scale = x.T @ d, x.T.abs() @ d.abs()
    _close(dy, want.T if transposed else want, scale.T if transposed else scale, ni, "dy")


# every gather order, a split sum, a column operand split ahead, the one-stage kernel
@pytest.mark.parametrize("ni,nk,nj", [(129, 65, 127), (300, 333, 65), (160, 5000, 136), (640, 200, 13001), (3077, 34, 3201)])
@pytest.mark.parametrize("transposed", [False, True])
@pytest.mark.parametrize("small,large", [(1e-37, 1e30), (1e-33, 1e-3), (1e-40, 1e33), (1e-5, 1e25)])
def test_operands_of_all_magnitudes(ni, nk, nj, transposed, small, large):
    """Operands whose second and third bf16 parts would be subnormal, subnormal ones, and large ones that are not split: the
    products are ordinary numbers and no less exact than others."""
    e = W.ex_matmul_t(ni, nj, nk) if transposed else W.ex_matmul(ni, nk, nj)
    args, df = W.make_inputs(e, ("normal", 0, 1), seed=nk)
    args[0] *= small
    args[1] *= large
    run = GpuRun(e, args, df)
    f = run.forward()
    dx, dy = run.backward()
    x, y, d = args[0].double(), args[1].double(), df.double()
    y = y.T if transposed else y
    subnormal = 2.0 ** -126                                     # (results may be subnormal themselves: a unit of 2^-149 per term)
    _close(f, x @ y, x.abs() @ y.abs() + nk * subnormal, nk, "forward")
    _close(dx, d @ y.T, d.abs() @ y.T.abs(), nj, "dx")
    want, scale = x.T @ d, x.T.abs() @ d.abs() + ni * subnormal
    _close(dy, want.T if transposed else want, scale.T if transposed else scale, ni, "dy")


@pytest.mark.parametrize("ni,nk,nj", [(600, 900, 2), (5, 1300, 700), (7, 4001, 130), (3000, 400, 3)])
def test_narrow_products(ni, nk, nj):
    """A side of a few rows or columns, as an output and as the summed side of the gradients."""
    test_matrix_products(ni, nk, nj, False)
    test_matrix_products(ni, nk, nj, True)


@pytest.mark.parametrize("ni,nk,nj", [(3077, 34, 3201), (3200, 64, 3072), (200, 17, 38000)])
def test_one_stage_contractions(ni, nk, nj):
    """At most 64 terms and enough tiles for the pipelined kernel: ragged edges in both directions, full and cut stages."""
    test_matrix_products(ni, nk, nj, False)
    test_matrix_products(ni, nk, nj, True)


@pytest.mark.parametrize("nb,nc,no,nt,nu", [(2, 64, 72, 130, 5), (3, 13, 65, 257, 3), (1, 20, 128, 64, 4)])
def test_strided_convolution(nb, nc, no, nt, nu):
    """Guards, several digits per group and strided stores (the residue classes of dx)."""
    e = W.conv1d(nb, nc, no, nt, nu)
    args, df = W.make_inputs(e, ("normal", 0, 1), seed=nt)
    run = GpuRun(e, args, df)
    f = run.forward()
    dx, dw = run.backward()

    def conv(x, w, d):
        x.requires_grad_(True), w.requires_grad_(True)
        out = torch.nn.functional.conv1d(x, w, stride=2)[:, :, :nt]
        return (out.detach(),) + torch.autograd.grad(out, (x, w), d)
    want = conv(args[0].double(), args[1].double(), df.double())
    scale = conv(args[0].double().abs(), args[1].double().abs(), df.double().abs())
    for got, w, s, n, what in zip((f, dx, dw), want, scale, (nc * nu, no * nu, nb * nt), ("forward", "dx", "dw")):
        _close(got, w, s, n, what)


# (rows, summed, columns): every gather order of the operand that is split ahead, ragged tiles and stages, with and without a split
@pytest.mark.parametrize("ni,nk,nj", [(700, 5003, 501), (5003, 501, 700), (640, 200, 13001)])
def test_columns_split_ahead(ni, nk, nj):
    for e in (W.ex_matmul(ni, nk, nj), W.ex_matmul_t(ni, nj, nk)):
        assert any("columns split ahead" in Plan(e).disassemble(w) for w in (-1, 0, 1))
    test_matrix_products(ni, nk, nj, False)
    test_matrix_products(ni, nk, nj, True)


@pytest.mark.parametrize("nb,nc,no,nt,nu", [(1, 3000, 512, 500, 3), (16, 96, 160, 1100, 5)])
def test_convolution_split_ahead(nb, nc, no, nt, nu):
    """A guarded operand split ahead, and one whose rows are windows."""
    assert "columns split ahead" in Plan(W.conv1d(nb, nc, no, nt, nu)).disassemble(-1)
    test_strided_convolution(nb, nc, no, nt, nu)


def test_split_ahead_without_room():
    """A workspace that holds all but the split operand gives the same result, as does a forward call without any."""
    e = W.conv1d(16, 96, 160, 1100, 5)
    args, df = W.make_inputs(e, ("normal", 0, 1), seed=5)
    run = GpuRun(e, args, df)
    f, grads = run.forward(), run.backward()
    run.plan.forward([a.data_ptr() for a in run.args], run.f.data_ptr(), torch.cuda.current_stream().cuda_stream)
    run.ws = run.ws[:-1]
    again = run.backward()
    scale = torch.nn.functional.conv1d(args[0].double().abs(), args[1].double().abs(), stride=2)[:, :, :1100]
    _close(run.f.cpu().numpy(), torch.from_numpy(f).double(), scale, 480, "forward")
    for a, b in zip(again, grads):
        assert float(abs(a - b).max()) <= 1e-5 * float(abs(b).max())


# a ragged tile, several stages and shares, a column operand split ahead, the one-stage kernel
@pytest.mark.parametrize("ni,nk,nj", [(130, 70, 140), (160, 5000, 136), (700, 5003, 501), (3077, 34, 3201)])
@pytest.mark.parametrize("transposed", [False, True])
def test_nan_rows_and_infinities(ni, nk, nj, transposed):
    """NaNs reach the outputs that read them and no others; sums with an infinity among other values, of either sign and of both."""
    e = W.ex_matmul_t(ni, nj, nk) if transposed else W.ex_matmul(ni, nk, nj)
    args, df = W.make_inputs(e, ("normal", 0, 1), seed=ni)
    x, y = args
    yt = y.T if transposed else y                               # summed x columns (a view)
    yt[yt.abs() < 1e-3] = 0.5
    x[3, nk // 2], x[ni - 1, 0], yt[nk - 1, nj - 2] = math.nan, math.nan, math.nan
    x[5, 7], x[6, 3], x[6, 9], x[ni // 2, nk - 2] = math.inf, math.inf, -math.inf, -math.inf
    yt[11, 17] = -math.inf
    f = torch.from_numpy(GpuRun(e, args, df).forward()).double()
    want = x.double() @ yt.double()
    assert torch.equal(f.isnan(), want.isnan())
    infinite = want.isinf()
    assert torch.equal(f[infinite], want[infinite])
    finite = want.isfinite()
    scale = x.double().abs() @ yt.double().abs()
    assert bool(((f - want).abs()[finite] <= 1e-5 * scale[finite]).all())


@pytest.mark.parametrize("ni,nk,nj", [(2000, 700, 1900), (8192, 64, 8192)])
def test_non_finite_operands_do_not_stall(ni, nk, nj):
    """An operand full of NaNs, as a diverged run has it, or one infinity: a small multiple of the time of ordinary values."""
    e = W.ex_matmul(ni, nk, nj)
    args, df = W.make_inputs(e, ("normal", 0, 1), seed=1)

    run = GpuRun(e, args, df)
    ordinary_x = run.args[0].clone()

    def time():
        best = math.inf
        for _ in range(4):
            start, stop = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            start.record()
            run.plan.forward([x.data_ptr() for x in run.args], run.f.data_ptr(), torch.cuda.current_stream().cuda_stream,
                             run.ws.data_ptr(), run.ws.numel())
            stop.record()
            torch.cuda.synchronize()
            best = min(best, start.elapsed_time(stop))
        return best
    ordinary = time()
    # (measured: 4 to 5 times; 60 to 300 times when every output was summed from its own terms)
    run.args[0].fill_(math.nan)
    assert time() <= 15 * ordinary
    run.args[0].copy_(ordinary_x)
    run.args[0].view(-1)[77:78].fill_(math.inf)
    assert time() <= 15 * ordinary


@pytest.mark.parametrize("nk,nj", [(70, 140), (33, 76000)])
def test_non_finite_operands(nk, nj):
    """Infinities and NaNs of the operands, and values beyond the bf16 range, give what the definition gives."""
    e = W.ex_matmul(130, nk, nj)
    args, df = W.make_inputs(e, ("normal", 0, 1), seed=3)
    x, y = args
    y[y.abs() < 1e-3] = 0.5
    x[3, 5], x[40, nk - 1], x[129, 0], x[77, 7] = math.inf, -math.inf, math.nan, 3.4028234e38
    y[7] = 0.25
    f = torch.from_numpy(GpuRun(e, args, df).forward())
    assert torch.equal(f[3], math.inf * torch.sign(y[5]))
    assert torch.equal(f[40], -math.inf * torch.sign(y[nk - 1]))
    assert bool(f[129].isnan().all())
    want = x.double() @ y.double()
    rows = [r for r in range(130) if r not in (3, 40, 129)]
    assert bool(((f.double() - want)[rows].abs() <= 1e-5 * (x.double().abs() @ y.double().abs())[rows]).all())
