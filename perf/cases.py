"""The work a program has this library do, as timed cases.

A case is one pass through the public entry points:

  eval      y = table(x): a query stream through a table laid out beforehand
  fit       a function becomes a table and is evaluated: design, vertex
            values, table build, evaluation (what a program does per function)
  table     a training step through one table: PWLFunction forward, then its
            backward with the gradients of x, the vertex values and the knots
  channels  the channel-wise learnable map: a training step (forward, then
            the gradients of x, knots and values) or an inference pass
  batch     a batch of independent functions: design, vertex values, index
            and evaluation of the concatenated queries

Inputs are seeded; exact() gives the results in 64 bits from plain torch and
numpy.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

import paper_1510_02975_gb300 as pwl

DTYPE = {"fp32": torch.float32, "bf16": torch.bfloat16, "fp16": torch.float16}

# the paper's three functions on their domains
FUNCS = {
    "gaussian": {"kind": "gaussian", "a": -4.0, "b": 4.0, "p": [1.0, 0.0, 1.0]},
    "lorentzian": {"kind": "lorentzian", "a": -10.0, "b": 10.0, "p": [1.0, 0.0, 1.0]},
    "bessel_j0": {"kind": "bessel_j0", "a": 0.0, "b": 50.0, "p": [1.0, 1.0]},
}


def listed():
    return [
        # the small plain workload: one 64-knot Gaussian table, 10^6 queries (launch and host latency)
        {"name": "eval_small", "what": "eval", "func": "gaussian", "intervals": 63, "queries": 10**6,
         "draw": "uniform", "values": "fp32", "io": "fp32"},
        # the plain workload at scale: the largest table, 2^28 queries clustered where the curvature is
        {"name": "eval_scale", "what": "eval", "func": "lorentzian", "intervals": 4096, "queries": 1 << 28,
         "draw": "normal", "values": "fp32", "io": "fp32"},
        # reduced precision end to end: 16-bit table, queries and results, a ragged count
        {"name": "eval_bf16", "what": "eval", "func": "bessel_j0", "intervals": 1024, "queries": (1 << 27) + 3,
         "draw": "uniform", "values": "bf16", "io": "bf16"},
        # a new function is approximated and used: everything from f to y
        {"name": "fit_j0", "what": "fit", "func": "bessel_j0", "intervals": 1024, "queries": 1 << 20,
         "draw": "uniform", "form": "project"},
        # one training step of a single learnable table on a minibatch with a ragged size
        {"name": "table_step_small", "what": "table", "func": "gaussian", "intervals": 256, "queries": 100003,
         "draw": "normal"},
        # the same on a large stream
        {"name": "table_step_large", "what": "table", "func": "bessel_j0", "intervals": 1024, "queries": 1 << 26,
         "draw": "uniform"},
        # the channel-wise differentiation workload, full size: [65536, 4096], 257 knots
        {"name": "channels_train_full", "what": "channels", "rows": 65536, "channels": 4096, "intervals": 256,
         "io": "fp32", "train": True},
        # its mixed-precision form on a smaller batch
        {"name": "channels_train_bf16", "what": "channels", "rows": 16384, "channels": 4096, "intervals": 256,
         "io": "bf16", "train": True},
        # a small layer of a learnable activation, odd sizes (rows, channels not multiples of a tile)
        {"name": "channels_train_small", "what": "channels", "rows": 1000, "channels": 200, "intervals": 31,
         "io": "fp32", "train": True},
        # serving the trained map in BF16: a forward pass, nothing recorded
        {"name": "channels_infer_bf16", "what": "channels", "rows": 4096, "channels": 1024, "intervals": 64,
         "io": "bf16", "train": False},
        # the batched workload: 4096 functions, FP32 integrands, 16 density cells per interval
        {"name": "batch_4096", "what": "batch", "functions": 4096, "precision": "fp32", "cells": 16,
         "form": "project", "q_hi": 10**6},
        # a few dozen functions at the default (FP64) precision and density
        {"name": "batch_40_fp64", "what": "batch", "functions": 40, "precision": "fp64", "cells": 0,
         "form": "project", "q_hi": 10**6},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random):
    what = rng.choice(["eval", "eval", "fit", "table", "table", "channels", "channels", "channels", "batch"])
    func = rng.choice(sorted(FUNCS))
    if what == "eval":
        io = rng.choice(["fp32", "fp32", "bf16", "fp16"])
        return {"what": what, "func": func, "intervals": _log_int(rng, 15, 4096),
                "queries": _log_int(rng, 10**3, 1 << 28), "draw": rng.choice(["uniform", "normal"]),
                "values": rng.choice(["fp32", "fp32", "bf16", "fp16"]), "io": io}
    if what == "fit":
        return {"what": what, "func": func, "intervals": _log_int(rng, 15, 4096),
                "queries": _log_int(rng, 10**4, 10**7), "draw": "uniform",
                "form": rng.choice(["interp", "project"])}
    if what == "table":
        return {"what": what, "func": func, "intervals": _log_int(rng, 15, 4096),
                "queries": _log_int(rng, 10**3, 1 << 27), "draw": rng.choice(["uniform", "normal"])}
    if what == "channels":
        channels = _log_int(rng, 16, 4096)
        rows = _log_int(rng, 64, 65536)
        return {"what": what, "rows": rows, "channels": channels, "intervals": _log_int(rng, 7, 512),
                "io": rng.choice(["fp32", "bf16"]), "train": rng.random() < 0.7}
    precision = rng.choice(["fp32", "fp64"])
    functions = _log_int(rng, 4, 4096) if precision == "fp32" else _log_int(rng, 4, 40)
    return {"what": what, "functions": functions, "precision": precision,
            "cells": 16 if precision == "fp32" else rng.choice([0, 16]),
            "form": rng.choice(["interp", "project"]), "q_hi": 10**6}


# ---- inputs ------------------------------------------------------------------
def _generator(seed, salt):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 16 + salt)
    return g


def _queries(case, seed):
    """FP32 queries uniform on the domain, or normal(0, 1.5) clipped to it."""
    f = FUNCS[case["func"]]
    g = _generator(seed, 1)
    if case["draw"] == "uniform":
        return torch.rand(case["queries"], generator=g, device="cuda").mul_(f["b"] - f["a"]).add_(f["a"])
    return torch.randn(case["queries"], generator=g, device="cuda").mul_(1.5).clamp_(f["a"], f["b"])


def _table_arrays(case, form="project"):
    """FP64 knots and vertex values of the case's function."""
    f = FUNCS[case["func"]]
    knots = _design(f, case["intervals"], 64 * case["intervals"])
    return knots, _values(f, knots, form)


def _channel_arrays(case, seed):
    """Knots and values [C, N+1] (FP32) of a learnable map initialised from
    the Gaussian's projection on [-8, 8], jittered per channel; x ~ N(0, 2^2)
    and the upstream gradient ~ N(0, 1) in the I/O type."""
    n, c, r = case["intervals"], case["channels"], case["rows"]
    f = {"kind": "gaussian", "a": -8.0, "b": 8.0, "p": [1.0, 0.0, 1.0]}
    k64 = _design(f, n, 64 * n)
    v64 = _values(f, k64, "project")
    g = _generator(seed, 2)
    h = float(torch.diff(k64).min())
    knots = k64.float().repeat(c, 1)
    knots[:, 1:-1] += (torch.rand(c, n - 1, generator=g, device="cuda") - 0.5) * (0.4 * h)
    values = v64.float().repeat(c, 1) + torch.randn(c, n + 1, generator=g, device="cuda") * 1e-3
    dt = DTYPE[case["io"]]
    x = torch.randn(r, c, generator=g, device="cuda").mul_(2.0).to(dt)
    gy = torch.randn(r, c, generator=g, device="cuda").to(dt)
    return knots, values, x, gy


def _batch_arrays(case, seed):
    """Functions cycling Gaussian / Lorentzian / J0 with log-uniform scales,
    knot counts uniform on 16..4096, query counts log-uniform on
    [1e3, q_hi], queries uniform on each domain, concatenated.  The counts
    depend on the case only; the scales and the queries on the seed."""
    shape, scale = random.Random(case["functions"]), random.Random(seed)
    funcs, n_int, n_q = [], [], []
    for i in range(case["functions"]):
        s = math.exp(scale.uniform(math.log(0.1), math.log(10.0)))
        if i % 3 == 0:
            funcs.append({"kind": "gaussian", "a": -4 * s, "b": 4 * s, "p": [1.0, 0.0, s]})
        elif i % 3 == 1:
            funcs.append({"kind": "lorentzian", "a": -10 * s, "b": 10 * s, "p": [1.0, 0.0, s]})
        else:
            funcs.append({"kind": "bessel_j0", "a": 0.0, "b": 50.0, "p": [1.0, scale.uniform(0.5, 5.0)]})
        n_int.append(shape.randint(15, 4095))
        n_q.append(_log_int(shape, 1e3, case["q_hi"]))
    offsets = [0]
    for n in n_q:
        offsets.append(offsets[-1] + n)
    x = torch.rand(offsets[-1], generator=_generator(seed, 3), device="cuda")
    counts = torch.tensor(n_q, device="cuda")
    a = torch.tensor([f["a"] for f in funcs], device="cuda", dtype=torch.float32)
    w = torch.tensor([f["b"] - f["a"] for f in funcs], device="cuda", dtype=torch.float32)
    x.mul_(torch.repeat_interleave(w, counts, output_size=offsets[-1]))
    x.add_(torch.repeat_interleave(a, counts, output_size=offsets[-1]))
    return funcs, n_int, offsets, x


def prepare(case, seed):
    what = case["what"]
    if what == "eval":
        knots, values = _table_arrays(case)
        x = _queries(case, seed).to(DTYPE[case["io"]])
        return {"case": case, "table": pwl.Table(knots, values, case["values"]), "x": x, "y": torch.empty_like(x)}
    if what == "fit":
        return {"case": case, "func": FUNCS[case["func"]], "x": _queries(case, seed)}
    if what == "table":
        knots, values = _table_arrays(case)
        x = _queries(case, seed).requires_grad_(True)
        gy = torch.randn(case["queries"], generator=_generator(seed, 4), device="cuda")
        return {"case": case, "table": pwl.Table(knots, values), "x": x, "gy": gy}
    if what == "channels":
        knots, values, x, gy = _channel_arrays(case, seed)
        if case["train"]:
            for t in (knots, values, x):
                t.requires_grad_(True)
        return {"case": case, "knots": knots, "values": values, "x": x, "gy": gy,
                "status": pwl.ChannelPWL.new_status()}
    funcs, n_int, offsets, x = _batch_arrays(case, seed)
    b = pwl.Batch(funcs, n_int, m_per_interval=case["cells"])
    b.plan(offsets)
    fp64 = case["precision"] == "fp64"
    return {"case": case, "batch": b, "x": x, "y": torch.empty_like(x),
            "knots": b.knots(copy=False) if fp64 else b.knots_fp32(copy=False),
            "values": b.values(copy=False) if fp64 else b.values_fp32(copy=False)}


# ---- one pass ----------------------------------------------------------------
def run(state):
    case = state["case"]
    what = case["what"]
    if what == "eval":
        return state["table"](state["x"], state["y"])
    if what == "fit":
        knots = pwl.design(state["func"], case["intervals"])
        values = pwl.project(state["func"], knots, case["form"])
        return {"knots": knots, "values": values, "y": pwl.Table(knots, values)(state["x"])}
    if what == "table":
        n1 = case["intervals"] + 1
        gv = torch.zeros(n1, device="cuda")
        gk = torch.zeros(n1, device="cuda")
        y = pwl.PWLFunction.apply(state["table"], state["x"], (gv, gk))
        (gx,) = torch.autograd.grad(y, state["x"], state["gy"])
        return {"y": y, "gx": gx, "g_values": gv, "g_knots": gk}
    if what == "channels":
        x, knots, values = state["x"], state["knots"], state["values"]
        if not case["train"]:
            with torch.no_grad():
                return pwl.ChannelPWL.apply(x, knots, values, 0, 0, state["status"])
        y = pwl.ChannelPWL.apply(x, knots, values, 0, 0, state["status"])
        gx, gk, gv = torch.autograd.grad(y, (x, knots, values), state["gy"])
        return {"y": y, "gx": gx, "g_knots": gk, "g_values": gv}
    b = state["batch"]
    b.design(case["precision"])
    b.project(case["form"], precision=case["precision"])
    b.build()
    b.eval(state["x"], state["y"])
    # the views end with the batch, what a program keeps of them is a copy
    return {"y": state["y"], "knots": state["knots"].clone(), "values": state["values"].clone()}


# ---- what a pass cannot do without --------------------------------------------
# FP operations of a density sample or a quadrature node (f or f'', the 2/5
# power, sums), of an evaluation (cell, lerp) and of a gradient element.
_SAMPLE, _EVAL, _GRAD = 40, 4, 12


def work(case):
    what = case["what"]
    if what == "eval":
        q, e = case["queries"], 4 if case["io"] == "fp32" else 2
        return {"bytes": 2 * e * q + 8 * case["intervals"], "flops": _EVAL * q}
    if what == "fit":
        n, q = case["intervals"], case["queries"]
        return {"bytes": 8 * q + 32 * n, "flops": (64 + 8) * n * _SAMPLE + _EVAL * q}
    if what == "table":
        q = case["queries"]
        return {"bytes": 20 * q + 24 * case["intervals"], "flops": (_EVAL + _GRAD) * q}
    if what == "channels":
        e = 4 if case["io"] == "fp32" else 2
        q = case["rows"] * case["channels"]
        params = 8 * case["channels"] * (case["intervals"] + 1)
        if not case["train"]:
            return {"bytes": 2 * e * q + params, "flops": _EVAL * q}
        return {"bytes": 5 * e * q + 3 * params, "flops": (_EVAL + _GRAD) * q}
    shape = random.Random(case["functions"])
    n = q = 0
    for _ in range(case["functions"]):
        n += shape.randint(15, 4095)
        q += _log_int(shape, 1e3, case["q_hi"])
    nodes = 8 if case["form"] == "project" else 1
    return {"bytes": 8 * q + 16 * n, "flops": n * ((case["cells"] or 64) + nodes) * _SAMPLE + _EVAL * q}


# ---- 64-bit results without the library -----------------------------------------
def _j01(z, z_max):
    """J0 and J1 of z in [0, z_max] from Bessel's integrals
    J0 = (2/pi) int_0^{pi/2} cos(z sin t) dt and
    J1 = (2/pi) int_0^{pi/2} sin t sin(z sin t) dt by the midpoint rule, whose
    error with m nodes is J_{4m}(z) (torch's own double-precision J0 and J1
    are 4e-7 off near z = 5)."""
    m = int((z_max + 60.0) / 4.0) + 1
    t = (torch.arange(m, device=z.device, dtype=torch.float64) + 0.5) * (0.5 * math.pi / m)
    s = torch.sin(t)[:, None]
    p = s * z.reshape(1, -1)
    return torch.cos(p).mean(0).reshape(z.shape), (s * torch.sin(p)).mean(0).reshape(z.shape)


def _f(f, x):
    p = f["p"]
    if f["kind"] == "gaussian":
        return p[0] * torch.exp(-0.5 * ((x - p[1]) / p[2]) ** 2)
    if f["kind"] == "lorentzian":
        return p[0] / (1.0 + ((x - p[1]) / p[2]) ** 2)
    return p[0] * _j01(p[1] * x, p[1] * f["b"])[0]


def _f2(f, x):
    p = f["p"]
    if f["kind"] == "gaussian":
        u2 = ((x - p[1]) / p[2]) ** 2
        return p[0] * (u2 - 1.0) / p[2] ** 2 * torch.exp(-0.5 * u2)
    if f["kind"] == "lorentzian":
        u2 = ((x - p[1]) / p[2]) ** 2
        return p[0] * (6.0 * u2 - 2.0) / (p[2] ** 2 * (1.0 + u2) ** 3)
    z = p[1] * x
    j0, j1 = _j01(z, p[1] * f["b"])
    return p[0] * p[1] ** 2 * (torch.where(z < 1e-8, torch.full_like(z, 0.5), j1 / z) - j0)


def _design(f, n, m):
    """Knots x_i with G(x_i) = i G(b) / n for the midpoint-rule cumulative G
    of |f''|^(2/5) on m uniform cells."""
    delta = (f["b"] - f["a"]) / m
    k = torch.arange(m, device="cuda", dtype=torch.float64)
    d = _f2(f, f["a"] + (k + 0.5) * delta).abs() ** 0.4
    G = torch.zeros(m + 1, device="cuda", dtype=torch.float64)
    torch.cumsum(d, 0, out=G[1:])
    G *= delta
    tau = torch.arange(1, n, device="cuda", dtype=torch.float64) * G[-1] / n
    c = (torch.searchsorted(G, tau, right=True) - 1).clamp_(0, m - 1)
    step = ((tau - G[c]) / d[c]).clamp_(0.0, delta)
    x = torch.empty(n + 1, device="cuda", dtype=torch.float64)
    x[0], x[n] = f["a"], f["b"]
    x[1:n] = f["a"] + c * delta + step
    return x


_GL_X, _GL_W = (v.tolist() for v in np.polynomial.legendre.leggauss(8))


def _hat_system(f, x):
    """Diagonal, upper coupling and load of the hat functions' Gram system."""
    h = torch.diff(x)
    mid, half = 0.5 * (x[:-1] + x[1:]), 0.5 * h
    left, right = torch.zeros_like(h), torch.zeros_like(h)
    t_all = torch.tensor(_GL_X, device=x.device, dtype=x.dtype)[:, None]
    for v, t, w in zip(_f(f, mid + half * t_all) * half, _GL_X, _GL_W):
        left += w * 0.5 * (1.0 - t) * v
        right += w * 0.5 * (1.0 + t) * v
    zero = torch.zeros(1, device=x.device, dtype=x.dtype)
    diag = (torch.cat([h, zero]) + torch.cat([zero, h])) / 3.0
    return diag, torch.cat([h / 6.0, zero]), torch.cat([left, zero]) + torch.cat([zero, right])


def _solve(systems):
    """Symmetric tridiagonal systems (diagonal, upper, load), padded to one
    [rows, systems] array and eliminated together (numpy, 64 bits)."""
    n = [s[0].numel() for s in systems]
    rows = max(n)
    D, U, B = np.ones((rows, len(n))), np.zeros((rows, len(n))), np.zeros((rows, len(n)))
    for i, s in enumerate(systems):
        D[:n[i], i], U[:n[i], i], B[:n[i], i] = (v.cpu().numpy() for v in s)
    C = np.zeros_like(U)
    for r in range(rows):
        piv = D[r] - (U[r - 1] * C[r - 1] if r else 0.0)
        C[r] = U[r] / piv
        B[r] = (B[r] - (U[r - 1] * B[r - 1] if r else 0.0)) / piv
    for r in range(rows - 2, -1, -1):
        B[r] -= C[r] * B[r + 1]
    return [torch.tensor(B[:n[i], i].copy(), device="cuda") for i in range(len(n))]


def _values(f, knots, form):
    return _f(f, knots) if form == "interp" else _solve([_hat_system(f, knots)])[0]


def _lerp(knots, values, x):
    """(interval, delta, y) of points x (64 bits, any shape whose leading
    dimensions match those of the tables)."""
    n = knots.shape[-1] - 1
    xc = torch.minimum(torch.maximum(x, knots[..., :1]), knots[..., -1:])
    i = torch.searchsorted(knots, xc.contiguous(), right=True).clamp_(1, n)
    x0, x1 = knots.gather(-1, i - 1), knots.gather(-1, i)
    v0, v1 = values.gather(-1, i - 1), values.gather(-1, i)
    delta = (xc - x0) / (x1 - x0)
    return i, delta, (v1 - v0) / (x1 - x0), (1.0 - delta) * v0 + delta * v1


def _gradients(knots, values, x, gy):
    """(y, gx, g_knots, g_values) of points x under the upstream gradient gy:
    outside the domain only the end values have a gradient."""
    i, delta, slope, y = _lerp(knots, values, x)
    left, right = x < knots[..., :1], x > knots[..., -1:]
    inside = ~(left | right)
    gx = torch.where(inside, gy * slope, torch.zeros_like(gy))
    ga, gb = gy * (1.0 - delta), gy * delta
    gv = torch.zeros_like(values).scatter_add_(-1, i - 1, ga).scatter_add_(-1, i, gb)
    zero = torch.zeros_like(ga)
    gk = torch.zeros_like(knots)
    gk.scatter_add_(-1, i - 1, torch.where(inside, -slope * ga, zero))
    gk.scatter_add_(-1, i, torch.where(inside, -slope * gb, zero))
    return y, gx, gk, gv


def exact(case, seed):
    what = case["what"]
    if what in ("eval", "table"):
        knots, values = _table_arrays(case)
        # a table holds its knots in FP32 and its values in their storage type
        knots = knots.float().double()
        values = values.float().to(DTYPE[case.get("values", "fp32")]).double()
        if what == "eval":
            x = _queries(case, seed).to(DTYPE[case["io"]])
            y = torch.empty(x.numel(), device="cuda", dtype=torch.float64)
            for q in range(0, x.numel(), 1 << 25):
                y[q:q + (1 << 25)] = _lerp(knots, values, x[q:q + (1 << 25)].double())[3]
            return y
        x = _queries(case, seed).double()
        gy = torch.randn(case["queries"], generator=_generator(seed, 4), device="cuda").double()
        y, gx, gk, gv = _gradients(knots, values, x, gy)
        return {"y": y, "gx": gx, "g_values": gv, "g_knots": gk}
    if what == "fit":
        knots, values = _table_arrays(case, case["form"])
        y = _lerp(knots.float().double(), values.float().double(), _queries(case, seed).double())[3]
        return {"knots": knots, "values": values, "y": y}
    if what == "channels":
        knots, values, x, gy = _channel_arrays(case, seed)
        knots, values = knots.double(), values.double()
        y = torch.empty(x.shape, device="cuda", dtype=torch.float64)
        gx, gk, gv = torch.empty_like(y), torch.empty_like(knots), torch.empty_like(values)
        for c in range(0, case["channels"], 256):
            s = slice(c, c + 256)
            xt = x[:, s].t().double().contiguous()
            if case["train"]:
                yt, gxt, gk[s], gv[s] = _gradients(knots[s], values[s], xt, gy[:, s].t().double().contiguous())
                gx[:, s] = gxt.t()
            else:
                yt = _lerp(knots[s], values[s], xt)[3]
            y[:, s] = yt.t()
        return {"y": y, "gx": gx, "g_knots": gk, "g_values": gv} if case["train"] else y
    funcs, n_int, offsets, x = _batch_arrays(case, seed)
    cells = case["cells"] or 64
    knots = [_design(f, n, cells * n) for f, n in zip(funcs, n_int)]
    if case["form"] == "interp":
        values = [_f(f, k) for f, k in zip(funcs, knots)]
    else:
        values = _solve([_hat_system(f, k) for f, k in zip(funcs, knots)])
    y = torch.empty(offsets[-1], device="cuda", dtype=torch.float64)
    for i, (k, v) in enumerate(zip(knots, values)):
        q = slice(offsets[i], offsets[i + 1])
        y[q] = _lerp(k.float().double(), v.float().double(), x[q].double())[3]
    return {"y": y, "knots": torch.cat(knots), "values": torch.cat(values)}
