"""The work that users of this library have it do, as measurable cases.

A user compiles an element-wise defined tensor expression once (a ``Plan``), keeps it with a workspace and calls it
with device (or pinned host) buffers: ``forward`` evaluates the expression, ``backward`` its derivatives with respect
to every argument.  A case is a family of expressions, its sizes and the entry point:

  step      forward, then backward with all gradients (a training step)
  forward   the value alone (inference)
  backward  the gradients alone
  saved     a step of a plan that reads the saved forward output in its backward pass
  noalloc   forward, then backward on the library's built-in scratch (callers that cannot allocate)
  host      one step on pinned host buffers, copies included

Families (sizes of the listed cases come from the configurations, tests and benchmark of this repository):

  intro           f_ij  = exp(-sum_k ((a_ik + b_jk)^2 c_ii + d_{i+k}^3))         sums, a diagonal and a shifted read
  shifted         f_ij  = exp(x_{i+j}) tanh(x_{2i+3j}) W_ii                      strided one-dimensional index maps
  nonunimodular   f_ijk = sin(x_{2i+j, j-k+n-1}) y_{3k}^2                        index map with masks in its gradient
  conv1d          f_bot = sum_cu w_ocu x_{b,c,2t+u}                              strided convolution
  matmul          f_ij  = sum_k x_ik y_kj                                        matrix product
  elementary      all elementary functions, a short sum, shared subexpressions  expressions outside the special forms
"""
from __future__ import annotations

import math

import torch

from paper_1711_01348_b200 import Plan
from workloads import configs as W


def listed():
    return [
        # the expression of the paper's introduction at its own size: a call is a handful of short launches
        dict(name="intro_64_step", family="intro", entry="step", ni=64, nj=64, nk=5),
        # the same small problem from a caller that cannot allocate a workspace, odd sizes
        dict(name="intro_203x157_noalloc", family="intro", entry="noalloc", ni=203, nj=157, nk=7),
        # the benchmark's workload: a training step on large square outputs
        dict(name="intro_8192_step", family="intro", entry="step", ni=8192, nj=8192, nk=32),
        # ragged rectangular sizes, the backward pass reads the saved output
        dict(name="intro_1301x2477_saved", family="intro", entry="saved", ni=1301, nj=2477, nk=21),
        # data that lives in host memory: copies in and out are part of the call
        dict(name="intro_2048_host", family="intro", entry="host", ni=2048, nj=2048, nk=16),
        # strided one-dimensional reads, large and at the small odd size of the tests
        dict(name="shifted_4096_step", family="shifted", entry="step", n=4096),
        dict(name="shifted_301_step", family="shifted", entry="step", n=301),
        # three-dimensional outputs with a masked gradient
        dict(name="nonunimodular_512_step", family="nonunimodular", entry="step", n=512),
        # strided convolution of a training step, full size; and inference on a ragged one with few channels
        dict(name="conv1d_256_step", family="conv1d", entry="step", nb=64, nc=256, no=256, nt=2048, nu=5),
        dict(name="conv1d_ragged_forward", family="conv1d", entry="forward", nb=7, nc=53, no=37, nt=701, nu=3),
        # plain matrix product with ragged sizes
        dict(name="matmul_1500_step", family="matmul", entry="step", ni=1500, nk=1100, nj=1333),
        # a general expression: every elementary function, division, negative powers
        dict(name="elementary_200003_step", family="elementary", entry="step", n=200003),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    family = rng.choice(["intro", "intro", "intro", "shifted", "nonunimodular", "conv1d", "conv1d", "matmul", "elementary"])
    entry = rng.choice(["step", "step", "forward", "backward"])
    c = dict(family=family, entry=entry)
    if family == "intro":
        c.update(ni=_log_int(rng, 64, 8192), nj=_log_int(rng, 64, 8192), nk=rng.randint(5, 32))
        c["entry"] = rng.choice(["step", "step", "forward", "backward", "saved", "host", "noalloc"])
        # the built-in scratch holds 32 MiB, one staged adjoint among it; pinned host buffers stay moderate
        if c["entry"] == "noalloc":
            c.update(ni=_log_int(rng, 64, 1500), nj=_log_int(rng, 64, 1500))
        elif c["entry"] == "host":
            c.update(ni=_log_int(rng, 64, 2048), nj=_log_int(rng, 64, 2048))
    elif family == "shifted":
        c.update(n=_log_int(rng, 301, 4096))
    elif family == "nonunimodular":
        c.update(n=_log_int(rng, 37, 512))
    elif family == "conv1d":
        c.update(nb=_log_int(rng, 3, 64), nc=_log_int(rng, 13, 256), no=_log_int(rng, 11, 256), nt=_log_int(rng, 70, 2048),
                 nu=rng.choice([3, 5]))
    elif family == "matmul":
        c.update(ni=_log_int(rng, 150, 4096), nk=_log_int(rng, 67, 4096), nj=_log_int(rng, 150, 4096))
    else:
        c.update(n=_log_int(rng, 300, 1000000))
    return c


def _expr(c):
    f = c["family"]
    if f == "intro":
        return W.intro(c["ni"], c["nj"], c["nk"]), ("uniform", -0.5, 0.5)
    if f == "shifted":
        return W.shifted(c["n"]), ("uniform", -1.0, 1.0)
    if f == "nonunimodular":
        return W.nonunimodular(c["n"]), ("normal", 0.0, 1.0)
    if f == "conv1d":
        return W.conv1d(c["nb"], c["nc"], c["no"], c["nt"], c["nu"]), ("normal", 0.0, 0.1)
    if f == "matmul":
        return W.ex_matmul(c["ni"], c["nk"], c["nj"]), ("normal", 0.0, 1.0)
    return W.ex_all_ops(c["n"]), ("uniform", -0.9, 0.9)


def prepare(case, seed):
    e, dist = _expr(case)
    entry = case["entry"]
    dev = torch.device("cuda")
    g = torch.Generator(device=dev)
    g.manual_seed(int(seed))
    args = []
    for shape in e.arg_shapes:
        if dist[0] == "uniform":
            args.append(torch.rand(shape, generator=g, device=dev) * (dist[2] - dist[1]) + dist[1])
        else:
            args.append(torch.randn(shape, generator=g, device=dev) * dist[2] + dist[1])
    df = torch.randn(e.out_shape, generator=g, device=dev)
    plan = Plan(e, saved_forward=entry == "saved")
    s = dict(plan=plan, entry=entry)
    if entry == "host":
        pinned = lambda t: t.cpu().pin_memory()
        s["args"], s["df"] = [pinned(t) for t in args], pinned(df)
        s["f"] = torch.empty(e.out_shape, pin_memory=True)
        s["dargs"] = [torch.empty(shape, pin_memory=True) for shape in e.arg_shapes]
        s["ws"] = torch.empty(plan.staging_bytes(), dtype=torch.uint8, device=dev)
        return s
    s["args"], s["df"] = args, df
    s["f"] = torch.empty(e.out_shape, device=dev)
    s["dargs"] = [torch.empty(shape, device=dev) for shape in e.arg_shapes]
    s["ws"] = torch.empty(max(256, plan.workspace_bytes()), dtype=torch.uint8, device=dev)
    return s


def run(state):
    s = state
    plan, entry, ws, f = s["plan"], s["entry"], s["ws"], s["f"]
    stream = torch.cuda.current_stream().cuda_stream
    args = [t.data_ptr() for t in s["args"]]
    dargs = [t.data_ptr() for t in s["dargs"]]
    df = s["df"].data_ptr()
    if entry == "host":
        plan.step_host(args, df, f.data_ptr(), dargs, ws.data_ptr(), ws.numel(), stream)
        return [f] + s["dargs"]
    if entry != "backward":
        plan.forward(args, f.data_ptr(), stream, ws.data_ptr(), ws.numel())
    if entry == "forward":
        return [f]
    if entry == "noalloc":
        plan.backward_noalloc(args, df, dargs, stream)
    else:
        # a plan compiled with saved_forward takes the forward output behind its arguments
        plan.backward(args + [f.data_ptr()] if entry == "saved" else args, df, dargs, ws.data_ptr(), ws.numel(), stream)
    return s["dargs"] if entry == "backward" else [f] + s["dargs"]


def work(case):
    """Every argument, df and f once each way they go; the operations of the definition, shared factors taken out of
    the sums (a multiplication or an addition 1, an elementary function 1)."""
    e, _ = _expr(case)
    c, f = case, case["family"]
    out = math.prod(e.out_shape)
    sizes = [math.prod(shape) for shape in e.arg_shapes]
    read = sum(sizes)
    if f == "intro":
        # only the diagonal of c is read
        read += c["ni"] - sizes[2]
        fwd = 2.0 * out * c["nk"] + 2.0 * out
        # G = df f, G b, G^T a, row sums
        bwd = 4.0 * out * c["nk"] + 3.0 * out
    elif f == "shifted":
        read += c["n"] - sizes[1]
        fwd, bwd = 2.0 * out, 7.0 * out
    elif f == "nonunimodular":
        fwd, bwd = 1.0 * out, 4.0 * out
    elif f == "conv1d":
        fwd = 2.0 * out * c["nc"] * c["nu"]
        bwd = 2.0 * fwd
    elif f == "matmul":
        fwd = 2.0 * out * c["nk"]
        bwd = 2.0 * fwd
    else:
        fwd, bwd = 40.0 * out, 80.0 * out
    entry = case["entry"]
    n_bytes = flops = 0.0
    if entry != "backward":
        n_bytes += 4.0 * (read + out)
        flops += fwd
    if entry != "forward":
        # arguments and df in, every gradient out
        n_bytes += 4.0 * (read + out + sum(sizes))
        flops += bwd
    return {"bytes": n_bytes, "flops": flops}


def tolerance(case):
    """Four times the largest error seen against the same expression in float64 (outputs and gradients, listed and
    drawn sizes): 7.7e-7 for the sums of products (a weight gradient over 131072 terms), 4.5e-7 for the gradients of
    intro, 4.5e-7 for the three elements of the elementary case that are sums over all outputs (taken wider: few
    elements, so one that nearly cancels weighs), 2.4e-7 for the others."""
    return {"rel": {"intro": 3e-6, "conv1d": 3e-6, "matmul": 3e-6, "elementary": 5e-6}.get(case["family"], 1e-6)}
