"""Cores of tile programs that are read step by step.  On the CPU the program that a plan lists is run point by point (two values, a sum)
in float64 and compared with the oracle, over random terms that couple the rows of one tensor with the rows of another; on the GPU
the kernels themselves, over as many of these terms as it takes to have every step, every kind of operand, both forms of the sum and a
factor outside.  Both compare the first rows of either tensor, which need the other one in full."""
import functools
import re

import numpy as np
import pytest

from oracle.oracle import Oracle, max_threads
from paper_1711_01348_b200 import Plan
from workloads.expr import Builder, unit

NESTED = 5000                   # from here on quotients of quotients
ROWS = 13                       # rows that are compared
SEEDS = 120
GPU_SEEDS = list(range(24)) + [34, 191, 207, 527, 1912, 2581]      # (with these every step is met)
FUNCTIONS = ["exp", "log", "sin", "cos", "tanh", "sinh", "cosh"]


# ---- random terms -----------------------------------------------------------------------------------------------------------------
def _sizes(seed):
    rng = np.random.default_rng(seed)
    return int(rng.integers(700, 1100)), int(rng.integers(500, 900)), int(rng.integers(8, 20))


def build(seed, ni=None, nj=None, tail=True):
    """f_ij = sum_k term, -(sum_k term) / 8 or f_i = sum_j sum_k term by turns; ni, nj: fewer rows of the same expression"""
    full = _sizes(seed)
    ni, nj, nk = ni or full[0], nj or full[1], full[2]
    summed = seed % 3 == 2
    shapes = {"x": [ni, nk], "y": [nj, nk], "z": [ni, nk], "w": [ni], "u": [nj], "v": [nk], "t": [ni, nj]}
    i, j, k = unit(3, (0, 1)), unit(3, (1, 1)), unit(3, (2, 1))
    rows = {"x": [i, k], "y": [j, k], "z": [i, k], "w": [i], "u": [j], "v": [k], "t": [i, j]}

    def grow(b, names):
        """one term: the same random numbers whatever the names are declared as"""
        rng = np.random.default_rng(1000 + seed)

        def leaf(*of):
            name = str(rng.choice(of))
            names.append(name)
            return b.load(name, rows[name]) if b else 0

        def wrap(a):
            how = rng.choice(["sq", "cube", "neg", "scale", "shift", "fn", "none", "none"])
            f = str(rng.choice(FUNCTIONS))
            if b is None:
                return a
            if how in ("sq", "cube"):
                return b.powi(a, 2 if how == "sq" else 3)
            if how == "neg":
                return b.un("neg", a)
            if how in ("scale", "shift"):
                return b.bin("mul" if how == "scale" else "add", a, b.const(-1.25 if how == "scale" else 1.5))
            if how == "fn":
                return b.un(f, b.bin("add", b.powi(a, 2), b.const(1.5)) if f == "log" else b.bin("mul", a, b.const(0.25)) if f in ("exp", "sinh", "cosh") else a)
            return a

        def join(a, c, ops=("add", "sub", "mul", "div")):
            op = str(rng.choice(ops))
            if rng.random() < 0.5:
                a, c = c, a
            return b.bin(op, a, c) if b else 0

        if seed >= NESTED:
            a, c, d = [leaf(n) for n in ("xyz", "zyw", "wxy", "xyw", "yxz", "uxy")[(seed - NESTED) // 3]]
            q = join(a, join(c, d, ("div",)), ("div",))
            return join(q, leaf("v"), ("mul",)) if seed % 2 else q
        t = wrap(join(leaf("x", "w"), leaf("y")) if rng.random() < 0.75 else join(leaf("x"), leaf("y", "u")))
        if rng.random() < 0.55:
            t = wrap(join(t, leaf("z", "w", "u", "v", "t")))
        if rng.random() < 0.3:
            t = join(t, wrap(join(leaf("z"), leaf("y"))))
        if rng.random() < 0.4:
            t = join(t, leaf("z", "v"), ("mul",))
        if rng.random() < 0.35:
            t = join(t, leaf("t", "w", "u"), ("mul",))
        return t

    names = []
    grow(None, names)
    used = sorted(set(names))
    b = Builder("core_%d" % seed, [ni] if summed else [ni, nj], 2 if summed else 1, used, [shapes[n] for n in used])
    s = b.sum(2, 0, nk - 1, grow(b, []))
    if summed:
        b.sum(1, 0, nj - 1, s)
    elif seed % 3 == 1 and tail:
        b.un("neg", b.bin("mul", s, b.const(0.125)))
    return b.done()


def _first(arrays, names, ni, nj):
    """the tensors of the expression with fewer rows"""
    cut = {"x": (ni,), "z": (ni,), "w": (ni,), "y": (nj,), "u": (nj,), "t": (ni, nj)}
    return [np.ascontiguousarray(a[tuple(slice(c) for c in cut.get(n, ()))]) for a, n in zip(arrays, names)]


@functools.lru_cache(maxsize=None)
def case(seed):
    """expression, inputs, df, and what the oracle has: f and gradients of the first rows with the scales of their terms"""
    e = build(seed)
    ni, nj, _ = _sizes(seed)
    rng = np.random.default_rng(2000 + seed)
    args = [rng.uniform(0.5, 1.5, s).astype(np.float32).astype(np.float64) for s in e.arg_shapes]
    df = rng.standard_normal(e.out_shape).astype(np.float32).astype(np.float64)
    want = {}
    for few_i in (True, False):
        n, m = (ROWS, nj) if few_i else (ni, ROWS)
        o = Oracle(build(seed, n, m))
        a = _first(args, e.arg_names, n, m)
        d = df[:n] if len(e.out_shape) == 1 else df[:n, :m]
        if few_i:
            f = o.forward(a, nthreads=max_threads())[0]
            # (the error of a sum is measured by its terms, also where something is computed from it)
            want["f"] = f, Oracle(build(seed, n, m, False)).forward(a, nthreads=max_threads())[1] * (0.125 if seed % 3 == 1 else 1)
        dx, terms = o.backward(a, np.ascontiguousarray(d), nthreads=max_threads())
        want.update((name, (g, s)) for name, g, s in zip(e.arg_names, dx, terms) if name in ("xzwt" if few_i else "yu"))
    return e, args, df, want


# ---- the listed program, run point by point ---------------------------------------------------------------------------------------
FN = {0: np.exp, 1: np.log, 2: np.sin, 3: np.cos, 4: np.tanh, 5: np.sinh, 6: np.cosh}


class Program:
    def __init__(self, text):
        head = text.split("\n", 1)[0]
        m = re.match(r"; tile program: (\d+) x (\d+) outputs( \(columns summed\))?, sums of (\d+)", head)
        self.p, self.q, self.l, self.q_sum = int(m[1]), int(m[2]), int(m[4]), bool(m[3])
        self.built = "(built)" in head
        self.loads, self.ops, self.core, self.steps = [], [], [], []
        for line in text.split("\n")[1:]:
            w = line.replace("=", " ").replace("+", " ").replace(",", " ").split() if "steps=" in line or "post=" in line else line.replace("=", " ").split()
            if line.startswith(";   load"):
                self.loads.append({"ptr": int(w[4]), "base": int(w[6]), "p": int(w[8]), "q": int(w[10]), "l": int(w[12])})
                assert w[14] == "0,0"
            elif line.startswith(";   operand"):
                self.ops.append((w[3], ("steps", int(w[5]), int(w[6])) if w[4] == "steps" else ("form", float(w[4]), int(w[6]), int(w[8]), int(w[10]))))
            elif line.startswith(";   core"):
                self.core.append((w[2], int(w[3]), int(w[4]), float(w[5])))
            elif line.startswith(";   step"):
                self.steps.append((w[3], int(w[4]), int(w[5]), float(w[6])))
            elif line.startswith(";   post"):
                self.post, self.tail = (int(w[2]), int(w[3])), (int(w[5]), int(w[6]))
                self.base, self.out_p, self.out_q = int(w[9]), int(w[11]), int(w[13])
                assert "of 1,1" in line

    def run(self, tensors, limit):
        """values of the outputs below the flat index `limit`: (flat indices, values); tensors: flat arrays by pointer slot"""
        p, q, l = np.arange(self.p), np.arange(self.q), np.arange(self.l)
        p = p[self.base + p * self.out_p < limit]
        if not self.q_sum:
            q = q[self.base + q * self.out_q < limit]
        P, Q, L = p[:, None, None], q[None, :, None], l[None, None, :]

        def load(i):
            d = self.loads[i]
            at = np.full((1, 1, 1), d["base"])
            for c, v in (("p", P), ("q", Q), ("l", L)):
                at = at + d[c] * v if d[c] else at
            assert at.min() >= 0 and at.max() < tensors[d["ptr"]].size
            return tensors[d["ptr"]][at]

        def program(at, n, total=None):
            x = y = None
            for op, a, b, imm in self.steps[at:at + n]:
                if op == "LD":
                    v = total if a < 0 else load(a)
                    x = v if b == 0 else x + v if b == 1 else x * v if b == 2 else (x + v) ** 2
                elif op == "PUSH":
                    y = x
                elif op == "FN":
                    x = x ** a if b == 7 else FN[b](x)
                else:
                    x = {"CONST": lambda: np.float64(imm), "NEG": lambda: -x, "SQR": lambda: x * x, "CUBE": lambda: x ** 3, "MULC": lambda: x * imm, "ADDC": lambda: x + imm,
                         "ADDY": lambda: y + x, "SUBY": lambda: y - x, "MULY": lambda: y * x, "DIVY": lambda: y / x}[op]()
            return x

        values = []
        for kind, o in self.ops:
            v = program(o[1], o[2]) if o[0] == "steps" else o[1] * load(o[2]) ** o[3] * (load(o[4]) if o[4] >= 0 else 1.0)
            v = np.asarray(v) * np.ones((1, 1, 1))
            # an operand varies with what its kind says, no more
            assert v.shape[0] == 1 or kind in ("ROW", "ROWC", "MAT"), kind
            assert v.shape[1] == 1 or kind in ("COL", "COLC", "MAT"), kind
            assert v.shape[2] == 1 or kind in ("ROW", "COL"), kind
            values.append(v)
        x = y = None
        total = 0.0
        for op, a, b, imm in self.core:
            o, o2 = (values[i] if i < len(values) else None for i in (a, b))
            if op == "ACC":
                total = total + (x * o if b else x)
            elif op == "PUSH":
                y = x
            elif op == "BINY":
                x = (y + x, y - x, y * x, y / x)[a]
            elif op == "FN":
                x = FN[a | b << 2](x)
            else:
                x = {"LD": lambda: o, "ADD": lambda: x + o, "SUB": lambda: x - o, "RSUB": lambda: o - x, "MUL": lambda: x * o, "FMA": lambda: x * o + o2, "SQR": lambda: x * x,
                     "CUBE": lambda: x ** 3, "NEG": lambda: -x, "MULC": lambda: x * imm, "ADDC": lambda: x + imm}[op]()
        total = (total * np.ones((len(p), len(q), len(l)))).sum(2, keepdims=True)
        if self.q_sum:
            if self.post[1]:
                total = total * program(*self.post)
            total = (total * np.ones((len(p), len(q), 1))).sum(1, keepdims=True)
        out = program(*self.tail, total=total) * np.ones((len(p), 1 if self.q_sum else len(q), 1))
        flat = np.broadcast_to(self.base + self.out_p * P + (0 if self.q_sum else self.out_q * Q), out.shape)
        keep = flat < limit
        return flat[keep], out[keep]

    def features(self):
        if self.built:
            return set()
        found = {op if op not in ("FN", "BINY") else "%s %d" % (op, a | b << 2) for op, a, b, _ in self.core}
        found |= {"ACC weighted" for op, a, b, _ in self.core if op == "ACC" and b}
        found |= {"operand " + kind for kind, _ in self.ops} | {"operand program" for _, o in self.ops if o[0] == "steps"}
        return found | ({"columns summed"} if self.q_sum else set()) | ({"factor outside"} if self.q_sum and self.post[1] else set())


EVERY = ({"LD", "ADD", "SUB", "RSUB", "MUL", "FMA", "SQR", "CUBE", "NEG", "MULC", "ADDC", "PUSH", "ACC", "ACC weighted", "columns summed", "factor outside", "operand program"}
         | {"BINY %d" % i for i in range(4)} | {"FN %d" % i for i in range(7)} | {"operand " + k for k in ("ROW", "COL", "ROWC", "COLC", "MAT")})


def _programs(plan, e):
    """tile programs without preparation of a plan: by -1 (forward), -2 - s (stages), index expressions"""
    found = {}
    for w in [-1] + [-2 - s for s in range(plan.num_stages())] + list(range(len(e.accesses))):
        text = plan.disassemble(w)
        if text.startswith("; tile program"):
            found[w] = Program(text)
    return found


def _emulate(seed):
    e, args, df, want = case(seed)
    plan = Plan(e)
    progs = _programs(plan, e)
    tensors = {i: a.reshape(-1) for i, a in enumerate(args)}
    tensors[len(args)] = df.reshape(-1)
    checked = 0
    for w, prog in progs.items():
        if any(d["ptr"] not in tensors for d in prog.loads):
            continue                                    # (reads a staged adjoint)
        name = "f" if w == -1 else e.arg_names[e.accesses[w].arg] if w >= 0 else None
        if name not in want or (w >= 0 and sum(a.arg == e.accesses[w].arg for a in e.accesses) != 1):
            continue
        g, scale = want[name]
        with np.errstate(all="ignore"):
            at, got = prog.run(tensors, g.size)
        ok = np.isfinite(g.reshape(-1)[at])
        err = np.abs(got - g.reshape(-1)[at])[ok]
        assert np.all(err <= 1e-6 * scale.reshape(-1)[at][ok] + 1e-9), (seed, w, err.max())
        checked += ok.any()
    return checked


@pytest.mark.parametrize("part", range(6))
def test_listed_programs_against_the_oracle(part):
    assert sum(_emulate(seed) for seed in [*range(part, SEEDS, 6), GPU_SEEDS[24 + part]]) >= 10


@pytest.mark.parametrize("seed", range(NESTED, NESTED + 18))
def test_listed_quotients_against_the_oracle(seed):
    _emulate(seed)


def test_every_step_is_met():
    found = set()
    for seed in GPU_SEEDS:
        for prog in _programs(Plan(build(seed)), build(seed)).values():
            found |= prog.features()
    assert EVERY <= found, sorted(EVERY - found)


@pytest.mark.gpu
@pytest.mark.parametrize("seed", GPU_SEEDS + list(range(NESTED, NESTED + 18, 3)))
def test_cores(seed):
    import torch
    from tests.gpu_util import GpuRun, assert_close
    e, args, df, want = case(seed)
    run = GpuRun(e, [torch.from_numpy(a).float() for a in args], torch.from_numpy(df).float())
    got = dict(zip(e.arg_names, run.backward()), f=run.forward())
    for name, (g, scale) in want.items():
        part = got[name][tuple(slice(n) for n in g.shape)]
        assert_close(part, g, scale, "%s %s" % (e.name, name), np.isfinite(g) & np.isfinite(scale))
