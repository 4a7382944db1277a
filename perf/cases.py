"""Timed cases of the homogenization library, each through its public Python entry points.

listed() names the cases, draw() gives more of the same ranges, prepare() makes what a
program holds before the call (microstructure, solver context, fields or network), run()
is one call and its outputs, work() the bytes and operations one call cannot do without,
exact() the same outputs from plain torch in float64.

Kinds of call:

product   Solver.apply: one matrix-free product (I + B) e or (I + B^T) e, the piece a
          program with its own Krylov method or time loop calls.
solve     Solver.solve: the local field and one column of the effective tensor.
tensor    Solver.solve_all: the full effective tensor, all unit loads together.
batch     Batch.solve: a sweep over many cells of uneven sizes.
predict   Net.forward: the warm-start network on one cell.
train     Net.gradients: loss and gradients of one training step of that network.

Solutions of the float32 solver with float64 refinement are returned in float32: they are
stopped at a tolerance, and a program that keeps many of them stores no more digits.
"""
import math

import numpy as np
import torch

from paper_1004_1122_gb300 import fh, microstructure, warmstart

# The default tolerance of Solver.solve and Solver.solve_all.
TOL = 1e-8
# Sweeps stop at the accuracy their effective tensors are compared to.
BATCH_TOL = 1e-7
MAX_ITER = 20000
# Largest number of node updates exact() spends on a solve (about 10 s of float64 FFTs).
EXACT_NODE_STEPS = 6e9


def listed():
    return [
        # The 81^2 single-disk cell: the smallest call in use, all launch latency.
        {"name": "product 81x81 f64", "kind": "product", "n0": 81, "n1": 81, "n2": 0, "precision": "fp64",
         "transpose": False},
        # The product of the 2187^2 benchmark cell.
        {"name": "product 2187x2187 f32", "kind": "product", "n0": 2187, "n1": 2187, "n2": 0, "precision": "fp32",
         "transpose": False},
        # The transposed product on a ragged 3-D box (a non-symmetric Krylov method).
        {"name": "product^T 63x135x105 f32", "kind": "product", "n0": 63, "n1": 135, "n2": 105, "precision": "fp32",
         "transpose": True},
        # One solve of the 81^2 cell at contrast 10 in float64.
        {"name": "solve 81x81 f64 cg", "kind": "solve", "n0": 81, "n1": 81, "n2": 0, "precision": "fp64",
         "method": "cg", "contrast": 10.0},
        # The 255^2 grid of the paper's model problem by BiCG (radix 17, products by A and A^T).
        {"name": "solve 255x255 f64 bicg", "kind": "solve", "n0": 255, "n1": 255, "n2": 0, "precision": "fp64",
         "method": "bicg", "contrast": 100.0},
        # An uneven mid-size image at high contrast.
        {"name": "solve 405x675 refined", "kind": "solve", "n0": 405, "n1": 675, "n2": 0, "precision": "fp32_refined",
         "method": "cg", "contrast": 1000.0},
        # The benchmark cell: a 2187^2 disk image at contrast 100.
        {"name": "solve 2187x2187 refined", "kind": "solve", "n0": 2187, "n1": 2187, "n2": 0,
         "precision": "fp32_refined", "method": "cg", "contrast": 100.0},
        # One load of a 135^3 cell, as training pairs of the warm start are made.
        {"name": "solve 135x135x135 refined", "kind": "solve", "n0": 135, "n1": 135, "n2": 135,
         "precision": "fp32_refined", "method": "cg", "contrast": 100.0},
        # The largest call: the tensor of a 243^3 cell at contrast 1000.
        {"name": "tensor 243x243x243 refined", "kind": "tensor", "n0": 243, "n1": 243, "n2": 243,
         "precision": "fp32_refined", "contrast": 1000.0},
        # A sweep over 40 cells of 81 to 729 nodes per axis, two loads each.
        {"name": "batch 40 cells", "kind": "batch", "cells": 40, "low": 81, "high": 729, "contrast": 1000.0},
        # Prediction on the full 135^3 grid.
        {"name": "predict 135x135x135", "kind": "predict", "n0": 135, "n1": 135, "n2": 135},
        # One training step on the smaller 81^3 grid.
        {"name": "train 81x81x81", "kind": "train", "n0": 81, "n1": 81, "n2": 81},
    ]


# ---------------------------------------------------------------------------
# drawn cases
# ---------------------------------------------------------------------------
def _smooth(n, primes):
    for p in primes:
        while n % p == 0:
            n //= p
    return n == 1


def _axis(rng, low, high, primes=(3, 5, 7)):
    """An axis length with the given prime factors, spread over the logarithm of its range."""
    want = math.exp(rng.uniform(math.log(low), math.log(high)))
    sizes = [n for n in range(low, high + 1) if _smooth(n, primes)]
    return min(sizes, key=lambda n: abs(math.log(n / want)))


def _primes(rng):
    # most grids are odd with small factors; some are even, or have a factor 11, 13 or 17
    return (3, 5, 7) if rng.random() < 0.75 else (2, 3, 5, 7, 11, 13, 17)


def _log(rng, low, high):
    return round(math.exp(rng.uniform(math.log(low), math.log(high))), 3)


def draw(rng):
    kind = rng.choice(["product", "product", "solve", "solve", "solve", "tensor", "batch", "predict", "train"])
    if kind == "product":
        d, pr = rng.choice([2, 2, 3]), _primes(rng)
        n = [_axis(rng, 45, 2187, pr) for _ in range(2)] if d == 2 else [_axis(rng, 21, 243, pr) for _ in range(3)]
        return {"kind": kind, "n0": n[0], "n1": n[1], "n2": n[2] if d == 3 else 0,
                "precision": rng.choice(["fp32", "fp64"]), "transpose": rng.random() < 0.3}
    if kind == "solve":
        d, pr = rng.choice([2, 2, 3]), _primes(rng)
        precision = rng.choice(["fp32_refined", "fp32_refined", "fp64"])
        method = rng.choice(["cg", "cg", "cg", "bicg", "fixed_point"]) if precision == "fp64" else "cg"
        if d == 2:
            top = 2187 if precision == "fp32_refined" else 405
            n = [_axis(rng, 81, top, pr) for _ in range(2)]
        else:
            n = [_axis(rng, 27, 189 if precision == "fp32_refined" else 63, pr) for _ in range(3)]
        return {"kind": kind, "n0": n[0], "n1": n[1], "n2": n[2] if d == 3 else 0, "precision": precision,
                "method": method, "contrast": _log(rng, 10.0, 20.0 if method == "fixed_point" else 1000.0)}
    if kind == "tensor":
        d = rng.choice([2, 3])
        n = [_axis(rng, 81, 1215) for _ in range(2)] if d == 2 else [_axis(rng, 27, 189) for _ in range(3)]
        return {"kind": kind, "n0": n[0], "n1": n[1], "n2": n[2] if d == 3 else 0, "precision": "fp32_refined",
                "contrast": _log(rng, 10.0, 1000.0)}
    if kind == "batch":
        low = _axis(rng, 27, 135)
        return {"kind": kind, "cells": rng.randint(6, 40), "low": low, "high": _axis(rng, 3 * low, 9 * low),
                "contrast": _log(rng, 10.0, 1000.0)}
    # grids of the network are multiples of 27
    n = [27 * rng.randint(1, 5) for _ in range(3)]
    return {"kind": kind, "n0": n[0], "n1": n[1], "n2": n[2]}


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _grid(case):
    return tuple(case[k] for k in ("n0", "n1", "n2") if case[k])


def inclusions(shape, fraction, rmin, rmax, rng):
    """Overlapping periodic disks or balls, radii uniform in [rmin, rmax], as many as
    the Boolean model needs for the volume fraction."""
    d = len(shape)
    img = np.zeros(shape, dtype=np.uint8)
    r = rng.uniform(rmin, rmax, size=4096)
    mean = float(np.mean(math.pi * r ** 2 if d == 2 else 4.0 / 3.0 * math.pi * r ** 3))
    count = max(1, int(round(-math.log(1.0 - fraction) * img.size / mean)))
    for _ in range(count):
        rad = rng.uniform(rmin, rmax)
        near, dist2 = [], 0.0
        for a, n in enumerate(shape):
            c = rng.uniform(0.0, n)
            reach = min(int(rad) + 1, (n - 1) // 2)
            at = np.arange(int(round(c)) - reach, int(round(c)) + reach + 1)
            near.append(np.mod(at, n))
            dist2 = dist2 + (((at - c) ** 2).reshape([-1 if b == a else 1 for b in range(d)]))
        box = np.ix_(*near)
        img[box] |= (dist2 <= rad * rad).astype(np.uint8)
    return img


def _cell(shape, rng):
    n = min(shape)
    if len(shape) == 2:
        return inclusions(shape, 0.4, max(2.0, n / 270), max(4.0, n / 55), rng)
    return inclusions(shape, 0.25, max(1.5, n / 27), max(2.5, n / 13), rng)


def _load(d, rng):
    e = rng.normal(size=d)
    return e / np.linalg.norm(e)


def _problem(case, seed):
    """(phase image, phase tensors, load) of a single-cell case."""
    rng = np.random.default_rng(seed)
    shape = _grid(case)
    phase = _cell(shape, rng)
    if case["kind"] == "product":
        contrast = 10.0 ** rng.uniform(1.0, 3.0)
    else:
        contrast = case["contrast"]
    return phase, microstructure.isotropic_table([1.0, contrast], len(shape)), _load(len(shape), rng)


def _field(case, seed):
    shape = _grid(case)
    g = torch.Generator(device="cuda").manual_seed(int(seed) + 17)
    dtype = torch.float64 if case["precision"] == "fp64" else torch.float32
    return torch.randn((len(shape),) + shape, generator=g, device="cuda", dtype=dtype)


def _batch_cells(case, seed):
    rng = np.random.default_rng(seed)
    # five sizes from the smallest to the largest cell; the cells cycle through them
    r = math.log(case["high"] / case["low"]) / 4.0
    sizes = [n for n in range(3, 2188) if _smooth(n, (3, 5, 7))]
    sizes = [min(sizes, key=lambda n: abs(math.log(n / (case["low"] * math.exp(r * k))))) for k in range(5)]
    phases, tables = [], []
    for c in range(case["cells"]):
        phases.append(_cell((sizes[c % 5],) * 2, rng))
        rho = math.exp(rng.uniform(math.log(min(10.0, case["contrast"])), math.log(case["contrast"])))
        tables.append(microstructure.isotropic_table([1.0, rho], 2))
    return phases, tables


def _net_input(case, seed):
    """(parameters, input, target): features of the size and scale the network sees
    (log-contrast, indicator and first-order response channels, unit-load targets)."""
    shape = _grid(case)
    g = torch.Generator(device="cuda").manual_seed(int(seed) + 29)
    params = warmstart.init_params(11, 3, int(seed) + 3)
    ind = (torch.rand(shape, generator=g, device="cuda") < 0.3).float()
    x = torch.cat([(0.6 * ind)[None], ind[None], 0.5 * torch.randn((9,) + shape, generator=g, device="cuda")])
    t = 0.5 * torch.randn((9,) + shape, generator=g, device="cuda")
    return params, x.contiguous(), t


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("product", "solve", "tensor"):
        phase, table, load = _problem(case, seed)
        state = {"case": case, "solver": fh.Solver(phase, table, precision=case["precision"]), "load": load}
        if kind == "product":
            state["e"] = _field(case, seed)
        return state
    if kind == "batch":
        phases, tables = _batch_cells(case, seed)
        return {"case": case, "batch": fh.Batch(phases, tables, nloads=2, precision="fp32_refined")}
    params, x, t = _net_input(case, seed)
    net = fh.Net(_grid(case), 11, 9)
    net.set_params(params)
    return {"case": case, "net": net, "x": x, "t": t}


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "product":
        return state["solver"].apply(state["e"], transpose=case["transpose"])
    if kind == "solve":
        field, column, _ = state["solver"].solve(state["load"], tol=TOL, method=case["method"], max_iter=MAX_ITER)
        if case["precision"] == "fp64":
            return {"field": field, "column": column}
        return {"field": field.float(), "column": column.astype(np.float32)}
    if kind == "tensor":
        tensor, _ = state["solver"].solve_all(tol=TOL, max_iter=MAX_ITER)
        return tensor.astype(np.float32)
    if kind == "batch":
        tensors, _, _, _ = state["batch"].solve(np.eye(2), tol=BATCH_TOL, max_iter=MAX_ITER)
        return tensors.astype(np.float32)
    if kind == "predict":
        return state["net"].forward(state["x"])
    loss, gradient = state["net"].gradients(state["x"], state["t"])
    return {"loss": loss, "gradient": gradient}


# ---------------------------------------------------------------------------
# work
# ---------------------------------------------------------------------------
def _product_flops(nodes, d):
    # d real forward and d real inverse transforms, the d x d products and the projection
    return nodes * (2 * d * 2.5 * math.log2(nodes) + 2 * d * d + 6 * d)


def _steps(contrast, method="cg"):
    """Iterations of a solve to TOL at this contrast (observed growth of CG on such cells)."""
    if method == "fixed_point":
        return 0.5 * contrast * math.log(2.0 / TOL)
    return 0.8 * contrast ** 0.4 * math.log(2.0 / TOL) * (2 if method == "bicg" else 1)


_IO = [(11, 16, 0), (16, 32, 1), (32, 48, 2), (48, 64, 3), (64, 48, 3), (48, 48, 2), (48, 32, 2), (32, 32, 1),
       (32, 16, 1), (16, 16, 0), (16, 9, 0)]


def work(case):
    kind = case["kind"]
    if kind == "batch":
        r = math.log(case["high"] / case["low"]) / 4.0
        nodes = [(case["low"] * math.exp(r * (c % 5))) ** 2 for c in range(case["cells"])]
        return {"bytes": sum(nodes), "flops": sum(2 * _steps(case["contrast"] ** 0.75) * _product_flops(n, 2) for n in nodes)}
    shape = _grid(case)
    nodes, d = math.prod(shape), len(shape)
    if kind == "product":
        s = 8 if case["precision"] == "fp64" else 4
        return {"bytes": nodes * (2 * d * s + 1), "flops": _product_flops(nodes, d)}
    if kind == "solve":
        return {"bytes": nodes * (1 + 8 * d), "flops": _steps(case["contrast"], case["method"]) * _product_flops(nodes, d)}
    if kind == "tensor":
        return {"bytes": nodes * d, "flops": d * _steps(case["contrast"]) * _product_flops(nodes, d)}
    params = sum(27 * i * o + o for i, o, _ in _IO)
    flops = sum(2.0 * 27 * i * o * nodes / 27 ** l for i, o, l in _IO)
    if kind == "predict":
        return {"bytes": 4 * (20 * nodes + params), "flops": flops}
    return {"bytes": 4 * (20 * nodes + 2 * params), "flops": 3 * flops}


# ---------------------------------------------------------------------------
# the same outputs in float64 from plain torch
# ---------------------------------------------------------------------------
class _Reference:
    """(I + B) and (I + B^T) for fields of shape (loads, d, N...) on the half spectrum."""

    def __init__(self, phase, table):
        shape = phase.shape
        self.shape, self.d = shape, len(shape)
        lam = np.array([t[0, 0] for t in table])
        self.l0 = 0.5 * (lam.min() + lam.max())
        ph = torch.from_numpy(phase.astype(np.int64)).cuda()
        self.delta = torch.from_numpy(lam).cuda()[ph] - self.l0
        xi, keep = [], True
        for a, n in enumerate(shape):
            k = torch.arange(n // 2 + 1 if a == self.d - 1 else n, device="cuda")
            k = torch.where(k <= n // 2, k, k - n)
            at = [-1 if b == a else 1 for b in range(self.d)]
            if n % 2 == 0:  # no Green operator at Nyquist frequencies of even axes
                keep = keep & (k != n // 2).reshape(at)
            xi.append(k.double().reshape(at))
        k2 = sum(x * x for x in xi)
        k2[(0,) * self.d] = 1.0
        self.xi, self.w = xi, torch.where(k2 > 0, 1.0 / (self.l0 * k2), k2) * keep
        self.w[(0,) * self.d] = 0.0

    def green(self, tau):
        axes = tuple(range(2, 2 + self.d))
        f = torch.fft.rfftn(tau, dim=axes)
        s = sum(f[:, a] * self.xi[a] for a in range(self.d)) * self.w
        return torch.fft.irfftn(torch.stack([s * x for x in self.xi], dim=1), s=self.shape, dim=axes)

    def apply(self, e, transpose=False):
        return e + self.delta * self.green(e) if transpose else e + self.green(self.delta * e)

    def solve(self, loads):
        """CG from e = E to a relative residual of 1e-12, all loads together."""
        dims = tuple(range(1, 2 + self.d))
        dot = lambda a, b: (a * b).sum(dim=dims, keepdim=True)  # noqa: E731
        e0 = torch.from_numpy(np.asarray(loads)).cuda().reshape((-1, self.d) + (1,) * self.d)
        e0 = e0.expand((e0.shape[0], self.d) + self.shape)
        x = e0.clone()
        r = e0 - self.apply(x)
        p, rr, stop = r.clone(), dot(r, r), 1e-24 * dot(e0, e0)
        for k in range(5000):
            if k % 10 == 0 and bool((rr <= stop).all()):
                break
            ap = self.apply(p)
            live = rr > stop
            alpha = torch.where(live, rr / torch.where(live, dot(p, ap), torch.ones_like(rr)), torch.zeros_like(rr))
            x += alpha * p
            r -= alpha * ap
            new = dot(r, r)
            p = r + torch.where(live, new / rr, torch.zeros_like(rr)) * p
            rr = torch.where(live, new, rr)
        return x

    def columns(self, x):
        """<L e> per load, shape (loads, d)."""
        return ((self.delta + self.l0) * x).flatten(2).mean(dim=2)


def _conv(x, w, b):
    O, C = w.shape[:2]
    y, t = 0.0, 0
    for dz in (1, 0, -1):
        for dy in (1, 0, -1):
            for dx in (1, 0, -1):
                y = y + w[:, :, t] @ torch.roll(x, (dz, dy, dx), (1, 2, 3)).reshape(C, -1)
                t += 1
    return (y + b[:, None]).reshape((O,) + x.shape[1:])


def _network(flat, x):
    """(output, parameter tensors) of the network; products use the weights rounded to bfloat16."""
    act = lambda z: torch.where(z > 0, z, 0.1 * z)  # noqa: E731
    pool = lambda a: torch.nn.functional.avg_pool3d(a[None], 3)[0]  # noqa: E731
    up = lambda a: a.repeat_interleave(3, 1).repeat_interleave(3, 2).repeat_interleave(3, 3)  # noqa: E731
    p, layers, at = torch.from_numpy(flat).cuda(), [], 0
    for i, o, _ in _IO:
        w = p[at:at + 27 * i * o].bfloat16().double().reshape(o, i, 27).requires_grad_(True)
        at += 27 * i * o
        b = p[at:at + o].double().requires_grad_(True)
        at += o
        layers.append((w, b))
    a = [act(_conv(x, *layers[0]))]
    for l in (1, 2, 3):
        a.append(act(_conv(pool(a[-1]), *layers[l])))
    u = a[3]
    for l in (2, 1, 0):
        v = up(act(_conv(u, *layers[8 - 2 * l]))) + a[l]
        u = act(_conv(v, *layers[9 - 2 * l]))
    return _conv(u, *layers[10]), [q for layer in layers for q in layer]


def exact(case, seed):
    kind = case["kind"]
    if kind == "product":
        phase, table, _ = _problem(case, seed)
        return _Reference(phase, table).apply(_field(case, seed).double()[None], case["transpose"])[0]
    if kind in ("solve", "tensor"):
        shape = _grid(case)
        d = len(shape)
        if math.prod(shape) * (d if kind == "tensor" else 1) * 1.5 * _steps(case["contrast"]) > EXACT_NODE_STEPS:
            return None
        phase, table, load = _problem(case, seed)
        ref = _Reference(phase, table)
        x = ref.solve(load[None] if kind == "solve" else np.eye(d))
        col = ref.columns(x)
        return {"field": x[0], "column": col[0]} if kind == "solve" else col.T.contiguous()
    if kind == "batch":
        phases, tables = _batch_cells(case, seed)
        out = []
        for phase, table in zip(phases, tables):
            ref = _Reference(phase, table)
            out.append(ref.columns(ref.solve(np.eye(2))).T)
        return torch.stack(out)
    params, x, t = _net_input(case, seed)
    with torch.set_grad_enabled(kind == "train"):
        y, leaves = _network(params, x.double())
        if kind == "predict":
            return y
        loss = ((y - t.double()) ** 2).mean()
        grads = torch.autograd.grad(loss, leaves)
    return {"loss": float(loss), "gradient": torch.cat([g.reshape(-1) for g in grads])}
