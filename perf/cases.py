"""Performance cases: the work a user of this library has it do, through its
public entry points, from the smallest call to the largest workload.

Kinds of case (each is one pass of ``run``):

stream   one elementwise operator on n float-float values (for add12 / mul12:
         n packed binary32 pairs).
dot      a dot product and the gradients of both vectors, through autograd
         (``api`` "autograd") or by the plain calls ("calls").
comp     compensated Sum2 and Dot2 of plain binary32 vectors.
gemv     a GEMV with k right-hand sides and its adjoint: the product and the
         gradient of X (``grad`` "x": A is constant data) or of A and X
         (``grad`` "all": A is a weight).
gemm     a matrix product ("forward") or the product with both adjoints
         ("train").
batch    many uneven instances in one plan, run by replaying its captured
         graph: dot and AXPY vectors ("dot_axpy") or matrices ("gemv"), stored
         back to back in one buffer (``packed``) or each from a 16-byte
         boundary.

Inputs follow the laws of ``paper_cs_0603115_gb300.inputs``: magnitudes
log-uniform over 2^-20 .. 2^20 with a tenth of the second operands cancelling
the first to about 30 bits, and ill-conditioned dot products.
"""
from __future__ import annotations

import math

import torch

import paper_cs_0603115_gb300 as ff
from paper_cs_0603115_gb300 import batch, inputs

DEV = "cuda"
OPS = ("add12", "mul12", "add", "add_accurate", "mul", "div", "sqrt", "axpy")
COND = 1e6


def listed():
    return [
        # the shortest stream of the paper's timing tables: one small vector
        # operation of an iteration, where the call itself is what costs
        {"name": "stream_add_4k", "kind": "stream", "op": "add", "n": 4096},
        # a vector of about a million values with an odd tail: the ordinary
        # elementwise size
        {"name": "stream_div_1m", "kind": "stream", "op": "div", "n": (1 << 20) + 3},
        # the benchmark's stream: arrays of 2 GiB
        {"name": "stream_mul_256m", "kind": "stream", "op": "mul", "n": 1 << 28},
        # an inner product of an iterative solver with its gradient, on a
        # vector of an ordinary length
        {"name": "dot_train_100k", "kind": "dot", "n": 100_003, "api": "calls"},
        # the benchmark's ill-conditioned dot product with its gradient
        {"name": "dot_train_64m", "kind": "dot", "n": 1 << 26, "api": "autograd"},
        # compensated reductions of binary32 data of an odd length
        {"name": "comp_3m", "kind": "comp", "n": 3_000_001},
        # a small dense layer or a small linear operator, one vector
        {"name": "gemv_train_small", "kind": "gemv", "m": 300, "n": 1000, "k": 1, "grad": "all"},
        # a layer of ragged size with a few right-hand sides
        {"name": "gemv_train_odd", "kind": "gemv", "m": 2001, "n": 3001, "k": 5, "grad": "all"},
        # the benchmark's matrix (8 GiB) with sixteen right-hand sides
        {"name": "gemv_32768_k16", "kind": "gemv", "m": 32768, "n": 32768, "k": 16, "grad": "x"},
        # a matrix product of a few hundred rows with both adjoints, no size a
        # multiple of a tile
        {"name": "gemm_train_500", "kind": "gemm", "m": 500, "n": 300, "k": 700, "mode": "train"},
        # the benchmark's matrix product
        {"name": "gemm_4096", "kind": "gemm", "m": 4096, "n": 4096, "k": 4096, "mode": "forward"},
        # a thousand uneven dot and AXPY instances stored back to back
        {"name": "batch_dot_axpy_1k", "kind": "batch", "mix": "dot_axpy", "count": 1024, "most": 1_000_000,
         "packed": True},
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(("stream", "stream", "dot", "comp", "gemv", "gemv", "gemm", "batch"))
    if kind == "stream":
        return {"kind": kind, "op": rng.choice(OPS), "n": _log_int(rng, 4096, 1 << 28)}
    if kind == "dot":
        return {"kind": kind, "n": _log_int(rng, 1000, 1 << 26), "api": rng.choice(("autograd", "calls"))}
    if kind == "comp":
        return {"kind": kind, "n": _log_int(rng, 10_000, 1 << 26)}
    if kind == "gemv":
        m, n = _log_int(rng, 64, 16384), _log_int(rng, 64, 16384)
        if rng.random() < 0.5:  # half of the row lengths are even
            n += n & 1
        return {"kind": kind, "m": m, "n": n, "k": _log_int(rng, 1, 64), "grad": rng.choice(("x", "all"))}
    if kind == "gemm":
        return {"kind": kind, "m": _log_int(rng, 64, 2600), "n": _log_int(rng, 64, 2600), "k": _log_int(rng, 16, 2600),
                "mode": rng.choice(("forward", "train"))}
    mix = rng.choice(("dot_axpy", "gemv"))
    if mix == "gemv":
        return {"kind": kind, "mix": mix, "count": _log_int(rng, 16, 512), "most": _log_int(rng, 200, 4096),
                "packed": rng.random() < 0.5}
    return {"kind": kind, "mix": mix, "count": _log_int(rng, 64, 1024), "most": _log_int(rng, 1000, 1_000_000),
            "packed": rng.random() < 0.5}


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _pair(seed, device=DEV):
    """One float-float scalar of magnitude about one on the device."""
    g = torch.Generator(device="cpu")
    g.manual_seed(seed)
    return inputs.to_ff(0.5 + torch.rand(1, generator=g, dtype=torch.float64))[0].to(device)


def _batch_sizes(case):
    """Instance sizes, the offsets of their arrays in one buffer per role, and
    the buffers' lengths: a property of the workload, the same for all inputs."""
    count, most = case["count"], case["most"]
    g = torch.Generator(device="cpu")
    g.manual_seed(31 * most + count)

    def log_sizes(lo):
        u = torch.rand(count, generator=g, dtype=torch.float64)
        return torch.round(lo * (most / lo) ** u).to(torch.int64).tolist()

    def offsets(sizes):
        at, out = 0, []
        for s in sizes:
            out.append(at)
            at += s if case["packed"] else s + (s & 1)
        return out, at

    if case["mix"] == "gemv":
        m, n = log_sizes(32), log_sizes(32)
        return {"m": m, "n": n, "a": offsets([p * q for p, q in zip(m, n)]), "x": offsets(n), "y": offsets(m)}
    n = log_sizes(100)
    kinds = [(batch.DOT, batch.AXPY)[i % 2] for i in torch.randperm(count, generator=g).tolist()]
    zs = offsets([s if k == batch.AXPY else 0 for s, k in zip(n, kinds)])
    return {"n": n, "kinds": kinds, "x": offsets(n), "z": zs}


def _batch_inputs(case, seed):
    sizes = _batch_sizes(case)
    if case["mix"] == "gemv":
        g = torch.Generator(device=DEV)
        g.manual_seed(seed)
        a = inputs.to_ff(inputs.loguniform_f64(sizes["a"][1], g, DEV))
        x = inputs.to_ff(inputs.loguniform_f64(sizes["x"][1], g, DEV))
        return sizes, a, x, None
    e = inputs.elementwise(sizes["x"][1], seed, device=DEV)
    alpha = _pair(seed, "cpu").tolist()
    return sizes, e.a, e.b, alpha


def _inputs(case, seed):
    kind = case["kind"]
    if kind == "stream":
        e = inputs.elementwise(case["n"], seed, device=DEV)
        if case["op"] in ("add12", "mul12"):
            return {"args": (e.ab,)}
        if case["op"] == "sqrt":
            return {"args": (e.a_sqrt,)}
        if case["op"] == "axpy":
            return {"args": (tuple(_pair(seed, "cpu").tolist()), e.a, e.b)}
        return {"args": (e.a, e.b)}
    if kind == "dot":
        g = inputs.ill_dot(case["n"], COND, seed, device=DEV)
        return {"x": g.x, "y": g.y, "dout": _pair(seed)}
    if kind == "comp":
        g = inputs.ill_dot_f32(case["n"], COND, seed, device=DEV)
        return {"x": g.x, "y": g.y}
    if kind == "gemv":
        g = inputs.gemv(case["m"], case["n"], case["k"], seed, device=DEV)
        return {"A": g.A, "X": g.X, "dY": g.dY}
    g = inputs.gemm(case["m"], case["n"], case["k"], seed, device=DEV)
    return {"A": g.A, "B": g.B, "dC": g.dC}


def prepare(case, seed):
    if case["kind"] == "batch":
        sizes, a, b, alpha = _batch_inputs(case, seed)
        specs = []
        if case["mix"] == "gemv":
            out = torch.zeros((sizes["y"][1], 2), dtype=torch.float32, device=DEV)
            outs = (out,)
            for m, n, at, xt, yt in zip(sizes["m"], sizes["n"], sizes["a"][0], sizes["x"][0], sizes["y"][0]):
                specs.append((batch.GEMV, a[at:at + m * n].view(m, n, 2), b[xt:xt + n], out[yt:yt + m], None))
        else:
            dots = torch.zeros((case["count"], 2), dtype=torch.float32, device=DEV)
            z = torch.zeros((max(sizes["z"][1], 1), 2), dtype=torch.float32, device=DEV)
            outs = (dots, z)
            for i, (n, kind, xt, zt) in enumerate(zip(sizes["n"], sizes["kinds"], sizes["x"][0], sizes["z"][0])):
                out = dots[i] if kind == batch.DOT else z[zt:zt + n]
                specs.append((kind, a[xt:xt + n], b[xt:xt + n], out, alpha if kind == batch.AXPY else None))
        plan = batch.BatchPlan(batch.make_instances(specs)).capture()
        return {"case": case, "plan": plan, "keep": (a, b), "outs": outs}
    state = _inputs(case, seed)
    state["case"] = case
    if case.get("api") == "autograd":
        state["x"].requires_grad_(True)
        state["y"].requires_grad_(True)
    return state


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "stream":
        return getattr(ff, case["op"])(*state["args"])
    if kind == "dot":
        x, y = state["x"], state["y"]
        if case["api"] == "autograd":
            d = ff.ffdot(x, y)
            dx, dy = torch.autograd.grad(d, (x, y), state["dout"])
            return {"d": d.detach(), "dx": dx, "dy": dy}
        d = ff.dot(x, y)
        dx, dy = ff.dot_backward(state["dout"], x, y)
        return {"d": d, "dx": dx, "dy": dy}
    if kind == "comp":
        return {"sum2": ff.sum2(state["x"]), "dot2": ff.dot2(state["x"], state["y"])}
    if kind == "gemv":
        A, X, dY = state["A"], state["X"], state["dY"]
        out = {"Y": ff.gemv(A, X), "dX": ff.gemv_t(A, dY)}
        if case["grad"] == "all":
            out["dA"] = ff.gemv_dA(dY, X)
        return out
    if kind == "gemm":
        A, B = state["A"], state["B"]
        out = {"C": ff.gemm(A, B)}
        if case["mode"] == "train":
            out["dA"] = ff.gemm(state["dC"], B, transb=True)
            out["dB"] = ff.gemm(A, state["dC"], transa=True)
        return out
    state["plan"].launch()
    return state["outs"]


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
# Binary32 operations of a float-float multiply and add (Mul22: 12 with a fused
# Mul12; Add22: 11 and a comparison), division and square root.
_MUL, _ADD, _DIV, _SQRT = 12, 12, 15, 15


def work(case):
    kind = case["kind"]
    if kind == "stream":
        n, op = case["n"], case["op"]
        arrays = 2 if op in ("add12", "mul12", "sqrt") else 3
        flops = {"add12": 6, "mul12": 3, "add": _ADD, "add_accurate": 20, "mul": _MUL, "div": _DIV, "sqrt": _SQRT,
                 "axpy": _MUL + _ADD}[op]
        return {"bytes": 8 * arrays * n, "flops": flops * n}
    if kind == "dot":
        n = case["n"]  # x and y read once, dx and dy written once
        return {"bytes": 32 * n, "flops": (3 * _MUL + _ADD) * n}
    if kind == "comp":
        n = case["n"]  # x and y read once
        return {"bytes": 8 * n, "flops": (7 + 11) * n}
    if kind == "gemv":
        m, n, k, full = case["m"], case["n"], case["k"], case["grad"] == "all"
        nbytes = 8 * (m * n * (2 if full else 1) + 2 * k * n + 2 * k * m)
        return {"bytes": nbytes, "flops": (_MUL + _ADD) * m * n * k * (3 if full else 2)}
    if kind == "gemm":
        m, n, k, train = case["m"], case["n"], case["k"], case["mode"] == "train"
        nbytes = 8 * ((m * k + k * n) * (2 if train else 1) + m * n * (2 if train else 1))
        return {"bytes": nbytes, "flops": (_MUL + _ADD) * m * n * k * (3 if train else 1)}
    sizes = _batch_sizes(case)
    if case["mix"] == "gemv":
        terms = sum(m * n for m, n in zip(sizes["m"], sizes["n"]))
        return {"bytes": 8 * (terms + sum(sizes["m"]) + sum(sizes["n"])), "flops": (_MUL + _ADD) * terms}
    nbytes = sum(n * (16 if k == batch.DOT else 24) for n, k in zip(sizes["n"], sizes["kinds"]))
    return {"bytes": nbytes, "flops": (_MUL + _ADD) * sum(sizes["n"])}


# ---------------------------------------------------------------------------
# the same outputs from 64-bit arithmetic
# ---------------------------------------------------------------------------
def _value(x):
    return x[..., 0].double() + x[..., 1].double()


def _split(v):
    """A binary64 result as (hi, lo): its binary32 rounding and the rest."""
    hi = v.float().double()
    return torch.stack([hi, v - hi], dim=-1)


def _exact_stream(op, args):
    if op in ("add12", "mul12"):
        a, b = args[0][:, 0].double(), args[0][:, 1].double()
        return a + b if op == "add12" else a * b
    if op == "axpy":
        alpha = float(args[0][0]) + float(args[0][1])
        return alpha * _value(args[1]) + _value(args[2])
    a = _value(args[0])
    if op == "sqrt":
        return a.sqrt()
    b = _value(args[1])
    return a * b if op == "mul" else a / b if op == "div" else a + b


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        sizes, a, b, alpha = _batch_inputs(case, seed)
        if case["mix"] == "gemv":
            out = torch.zeros(sizes["y"][1], dtype=torch.float64, device=DEV)
            for m, n, at, xt, yt in zip(sizes["m"], sizes["n"], sizes["a"][0], sizes["x"][0], sizes["y"][0]):
                out[yt:yt + m] = _value(a[at:at + m * n]).view(m, n) @ _value(b[xt:xt + n])
            return (_split(out),)
        dots = torch.zeros(case["count"], dtype=torch.float64, device=DEV)
        z = torch.zeros(max(sizes["z"][1], 1), dtype=torch.float64, device=DEV)
        al = alpha[0] + alpha[1]
        for i, (n, k, xt, zt) in enumerate(zip(sizes["n"], sizes["kinds"], sizes["x"][0], sizes["z"][0])):
            x, y = _value(a[xt:xt + n]), _value(b[xt:xt + n])
            if k == batch.DOT:
                dots[i] = (x * y).sum()
            else:
                z[zt:zt + n] = al * x + y
        return _split(dots), _split(z)
    s = _inputs(case, seed)
    if kind == "stream":
        return _split(_exact_stream(case["op"], s["args"]))
    if kind == "dot":
        x, y, d = _value(s["x"]), _value(s["y"]), _value(s["dout"])
        return {"d": _split((x * y).sum()), "dx": _split(d * y), "dy": _split(d * x)}
    if kind == "comp":
        x, y = s["x"].double(), s["y"].double()
        return {"sum2": _split(x.sum()), "dot2": _split((x * y).sum())}
    if kind == "gemv":
        A, X, dY = _value(s["A"]), _value(s["X"]), _value(s["dY"])
        out = {"Y": _split(X @ A.t()), "dX": _split(dY @ A)}
        if case["grad"] == "all":
            out["dA"] = _split(dY.t() @ X)
        return out
    A, B = _value(s["A"]), _value(s["B"])
    out = {"C": _split(A @ B)}
    if case["mode"] == "train":
        dC = _value(s["dC"])
        out["dA"], out["dB"] = _split(dC @ B.t()), _split(A.t() @ dC)
    return out
