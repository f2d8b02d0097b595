"""Performance cases of the library: the calls a user makes, with their inputs, minimal work and 64-bit results.

A case is a dict of plain values.  ``kind`` names the entry points of one pass:

  step     autograd: reduce_by_index (+, hist0), reduce (+) and scan (+) of the same values, and their gradients
  hist     reduce_by_index forward (with residuals) and vjp of one operator, caller-held buffers
  scan     inclusive scan forward and vjp of one operator, caller-held buffers
  reduce   reduce forward and vjp of one operator, caller-held buffers
  rows     tuple scan over rows of independent blocks, forward and vjp
  vscan    vectorised scan over rows of d columns, forward and vjp
  batched  many (reduce_by_index -> +-scan -> sum) instances: the captured forward and backward graphs

``op``, ``dtype`` ("f32", "f64"), ``n`` (elements or rows), ``m`` (bins), ``k`` (blocks), ``d`` (columns) and
``count`` (instances) complete it.  Inputs follow the workloads of ``synth.py`` and of ``bench.py``, drawn on the
device from the seed.  Two differ, because the results would otherwise say little: reduce_by_index products take
``mul_wc``'s values (ln v ~ U(-delta, delta), delta = 10 / sqrt(n / m)) with about one zero in two bins, so that
bins without, with one and with several zeros all occur and nothing underflows; fp64 product scans and reduces take
delta = 10 / sqrt(n).
"""
import math
from types import SimpleNamespace

import numpy as np
import torch

from paper_2310_03568_gb300 import adcomb, autograd, batched

DTYPE = {"f32": torch.float32, "f64": torch.float64}
SIZE = {"f32": 4, "f64": 8}
Q = {"mm2": 2, "mm3": 3}
MOST_BYTES = 4.8e9  # of the largest listed case


def listed():
    return [
        # The smallest workload of the benchmark: a training step's worth of tiny calls through autograd, where
        # launches and host time are what a user waits for.
        {"name": "step_small", "kind": "step", "dtype": "f32", "n": 100_000, "m": 1000},
        # The headline workload (n = 50M): arg-max into few bins (private tables), ...
        {"name": "hist_max_401", "kind": "hist", "op": "max", "dtype": "f32", "n": 50_000_000, "m": 401},
        # ... products with zero counting into a table that fills a block's shared memory, ...
        {"name": "hist_mul_50k", "kind": "hist", "op": "mul", "dtype": "f32", "n": 50_000_000, "m": 50_000},
        # ... and arg-min into ten million bins (a table far beyond shared memory).
        {"name": "hist_min_10m", "kind": "hist", "op": "min", "dtype": "f32", "n": 50_000_000, "m": 10_000_000},
        # The general (non-commutative) reduce_by_index.
        {"name": "hist_lin_1000", "kind": "hist", "op": "lin", "dtype": "f32", "n": 10_000_000, "m": 1000},
        # Prefix sums and linear recurrences over the largest arrays.
        {"name": "scan_add_100m", "kind": "scan", "op": "add", "dtype": "f32", "n": 100_000_000},
        {"name": "scan_lin_100m", "kind": "scan", "op": "lin", "dtype": "f32", "n": 100_000_000},
        # The double-precision run of the same family.
        {"name": "scan_mul_f64_10m", "kind": "scan", "op": "mul", "dtype": "f64", "n": 10_000_000},
        # The general scan over 2x2 matrix products, a ragged size.
        {"name": "scan_mm2_10m", "kind": "scan", "op": "mm2", "dtype": "f32", "n": 9_999_991},
        # Reduction with arg-max tracking, a ragged size.
        {"name": "reduce_max_100m", "kind": "reduce", "op": "max", "dtype": "f32", "n": 99_999_989},
        # Row scans of tuples of 16 sumOfProd blocks, an ordinary ragged size.
        {"name": "rows_sop16_1m", "kind": "rows", "op": "sop", "k": 16, "dtype": "f32", "n": 1_000_003},
        # Batched autograd: a quarter of the 4096-instance workload, replayed graphs.
        {"name": "batched_1024", "kind": "batched", "dtype": "f32", "count": 1024},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    while True:
        kind = rng.choice(["step", "hist", "hist", "hist", "scan", "scan", "scan", "reduce", "rows", "vscan", "batched"])
        dtype = rng.choice(["f32", "f32", "f32", "f64"])
        if kind == "step":
            c = {"kind": kind, "dtype": dtype, "n": _log(rng, 1000, 1_000_000), "m": _log(rng, 31, 10_000)}
        elif kind == "hist":
            op = rng.choice(["add", "mul", "min", "max", "lin"])
            n = _log(rng, 1000, 10_000_000 if op == "lin" else 50_000_000)
            m = _log(rng, 31, 2000 if op == "lin" else 10_000_000)
            # The rounding error of an fp32 product grows with its length whatever the order: at most 1e4 values a bin.
            if op == "mul" and dtype == "f32" and n > 10_000 * m:
                m = -(-n // 10_000)
            c = {"kind": kind, "op": op, "dtype": dtype, "n": n, "m": m}
        elif kind == "scan":
            op = rng.choice(["add", "mul", "max", "lin", "sop", "mm2", "mm3"])
            c = {"kind": kind, "op": op, "dtype": dtype, "n": _log(rng, 1000, 10_000_000 if op[:2] == "mm" else 100_000_000)}
        elif kind == "reduce":
            op = rng.choice(["add", "max", "lin"] if dtype == "f32" else ["add", "mul", "max", "lin"])
            c = {"kind": kind, "op": op, "dtype": dtype, "n": _log(rng, 1000, 100_000_000)}
        elif kind == "rows":
            c = {"kind": kind, "op": rng.choice(["lin", "sop"]), "k": rng.randint(2, 16), "dtype": dtype, "n": _log(rng, 1000, 2_000_000)}
        elif kind == "vscan":
            c = {"kind": kind, "op": rng.choice(["add", "max"]), "d": rng.randint(2, 64), "dtype": dtype, "n": _log(rng, 1000, 2_000_000)}
        else:
            c = {"kind": kind, "dtype": "f32", "count": _log(rng, 16, 1024)}
        if work(c)["bytes"] <= MOST_BYTES:
            return c


def _width(case):
    """Scalars of one element of the case's arrays."""
    op = case.get("op", "add")
    w = {"lin": 2, "sop": 2, "mm2": 4, "mm3": 9}.get(op, 1)
    return w * case.get("k", case.get("d", 1))


def work(case):
    """Bytes each call of a pass cannot do without (inputs read once, outputs written once) and its arithmetic."""
    kind, op = case["kind"], case.get("op", "add")
    if kind == "batched":
        ns, ms, ops = _instances(case)
        n, m, n_add = float(ns.sum()), float(ms.sum()), float(ns[ops == 0].sum())
        return {"bytes": 8 * n + 8 * m + 4 * n + 4 * n_add + 4 * m, "flops": n + 2 * m + n_add}
    s, n = SIZE[case["dtype"]], float(case["n"])
    e = s * _width(case)
    if kind == "step":
        m = float(case["m"])
        # forward: keys, values, hist0 -> hist; values -> sum; values -> scan;  vjp: keys, histbar -> vbar, hist0bar;
        # broadcast; reverse scan; the three value gradients added
        return {"bytes": (4 + s) * n + 2 * s * m + s * n + 2 * s * n + (4 + s) * n + 2 * s * m + s * n + 2 * s * n + 4 * s * n, "flops": 6 * n}
    if kind == "hist":
        m = float(case["m"])
        fwd = (4 + e) * n + e * m
        vjp = {"add": 4 * n + e * n + e * m, "mul": (4 + 2 * e) * n + 2 * e * m, "min": e * n + (e + 4) * m,
               "max": e * n + (e + 4) * m, "lin": (4 + 2 * e) * n + e * m}[op]
        return {"bytes": fwd + vjp, "flops": (10 if op == "lin" else 3) * n}
    if kind == "reduce":
        vjp = {"add": e, "max": e, "mul": 2 * e, "lin": 2 * e}[op]
        return {"bytes": (e + vjp) * n, "flops": (10 if op == "lin" else 2) * n}
    vjp = {"add": 2, "max": 3}.get(op, 4)
    q = Q.get(op, 1)
    return {"bytes": (2 + vjp) * e * n, "flops": {"lin": 10.0, "sop": 10.0}.get(op, 6.0 * q ** 3) * n * _width(case) / ({"lin": 2, "sop": 2}.get(op, q * q))}


# ------------------------------------------------------------------ inputs --
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _uniform(g, shape, lo, hi, dt):
    return torch.rand(shape, generator=g, device="cuda", dtype=dt).mul_(hi - lo).add_(lo)


def _normal(g, shape, dt):
    return torch.randn(shape, generator=g, device="cuda", dtype=dt)


def _keys(g, n, m):
    return torch.randint(0, m, (n,), generator=g, device="cuda", dtype=torch.int32)


def _levels(g, n, dt):
    """1024 distinct levels: ties are common."""
    return (torch.randint(0, 1024, (n,), generator=g, device="cuda", dtype=torch.int32) - 512).to(dt) / 64.0


def _values(g, kind, op, n, m, dt):
    if op == "add":
        return _uniform(g, n, 0.0 if kind == "reduce" else -1.0, 1.0, dt)
    if op in ("min", "max"):
        return _normal(g, n, dt) if kind == "scan" else _levels(g, n, dt)
    if op == "mul":
        if kind == "scan" and dt == torch.float32:  # scan_spec: 0.1% exact zeros
            v = _uniform(g, n, 0.9, 1.1, dt)
            v[torch.rand(n, generator=g, device="cuda") < 0.001] = 0
            return v
        delta = 10.0 / math.sqrt(max(n / m, 1.0))
        v = _uniform(g, n, -delta, delta, dt).exp_()
        if kind == "hist":
            v[torch.rand(n, generator=g, device="cuda") < min(0.01, 0.5 * m / n)] = 0
        return v
    if op == "lin":
        return torch.stack([_normal(g, n, dt), _uniform(g, n, 0.95, 1.05, dt)], dim=1)
    if op == "sop":
        return _uniform(g, (n, 2), -1.0, 1.0, dt)
    q = Q[op]
    return _uniform(g, (n, q * q), -1.0, 1.0, dt).div_(math.sqrt(q))


def _instances(case):
    """Sizes and operators of the batched instances (host; part of the case, not of the seed)."""
    r = np.random.default_rng(4)
    c = int(case["count"])
    ns = np.round(np.exp(r.uniform(np.log(1e3), np.log(1e6), c))).astype(np.int64)
    ms = np.round(np.exp(r.uniform(np.log(64), np.log(65536), c))).astype(np.int64)
    return ns, ms, np.where(r.random(c) < 0.5, 0, 1).astype(np.int32)  # 0: +, 1: max


def _batched_inputs(case, seed):
    ns, ms, ops = _instances(case)
    desc = batched.make_table(ns, ms, ops)
    total = int((desc["val_off"] + desc["n"]).max())
    g = _gen(seed)
    inst = torch.repeat_interleave(torch.arange(len(ns), device="cuda"),
                                   torch.from_numpy(np.diff(np.append(desc["val_off"], total))).cuda())
    pos = torch.arange(total, device="cuda") - torch.from_numpy(desc["val_off"].copy()).cuda()[inst]
    m = torch.from_numpy(ms).cuda()[inst]
    keys = (torch.rand(total, generator=g, device="cuda", dtype=torch.float64) * m).to(torch.int32)
    keys = torch.minimum(keys, (m - 1).to(torch.int32))
    pad = pos >= torch.from_numpy(ns).cuda()[inst]
    keys[pad] = -1  # between instances: never read
    vals = _uniform(g, total, -1.0, 1.0, torch.float32)
    vals[pad] = 0
    return desc, keys, vals, inst


def _inputs(case, seed):
    kind, op, dt, n = case["kind"], case.get("op", "add"), DTYPE[case["dtype"]], case["n"]
    g = _gen(seed)
    s = SimpleNamespace(kind=kind, op=op, n=n, m=case.get("m", 0))
    if kind == "step":
        s.keys, s.x, s.h0 = _keys(g, n, s.m), _uniform(g, n, -1.0, 1.0, dt), _uniform(g, s.m, -1.0, 1.0, dt)
        s.hb, s.rb, s.sb = _normal(g, s.m, dt), _normal(g, 1, dt).reshape(()), _normal(g, n, dt)
    elif kind == "hist":
        s.keys, s.x = _keys(g, n, s.m), _values(g, kind, op, n, s.m, dt)
        s.hb = _normal(g, (s.m, 2) if op == "lin" else s.m, dt)
    elif kind in ("rows", "vscan"):
        w = _width(case)
        if op == "lin":
            s.x = _values(g, kind, op, n * case["k"], 1, dt).reshape(n, w)
        else:
            s.x = _uniform(g, (n, w), -1.0, 1.0, dt)
        s.yb = _normal(g, (n, w), dt)
        s.ops = [op] * case.get("k", 0)
    else:
        s.x = _values(g, kind, op, n, 1, dt)
        s.yb = _normal(g, tuple(s.x.shape) if kind == "scan" else (s.x.shape[1:] or (1,)), dt)
    return s


def prepare(case, seed):
    if case["kind"] == "batched":
        desc, keys, vals, _ = _batched_inputs(case, seed)
        p = batched.BatchedHistScan(desc, keys, vals)
        p.hist.zero_()  # the bins between instances are never written
        p.scan.zero_()
        p.capture()
        return SimpleNamespace(kind="batched", problem=p)
    s = _inputs(case, seed)
    if s.kind == "step":
        s.x.requires_grad_(True)
        s.h0.requires_grad_(True)
        return s
    # output and residual buffers, held as a training loop holds them
    dev, dt = s.x.device, s.x.dtype
    s.xb = torch.empty_like(s.x)
    if s.kind == "hist":
        s.y = torch.empty_like(s.hb)
        s.saved = torch.empty(max(adcomb.saved_bytes("hist", s.op, dt, s.n, s.m), 16), dtype=torch.uint8, device=dev)
    elif s.kind == "reduce":
        s.y = torch.empty_like(s.yb)
        s.saved = torch.empty(max(adcomb.saved_bytes("reduce", s.op, dt, s.n), 16), dtype=torch.uint8, device=dev)
    else:
        s.y = torch.empty_like(s.x)
    return s


# --------------------------------------------------------------------- run --
def run(s):
    if s.kind == "step":
        h = autograd.reduce_by_index(s.x, s.keys, s.m, "add", s.h0)
        r = autograd.reduce(s.x, "add")
        y = autograd.scan(s.x, "add")
        gx, gh0 = torch.autograd.grad([h, r, y], [s.x, s.h0], [s.hb, s.rb, s.sb])
        return {"hist": h, "sum": r, "scan": y, "xbar": gx, "hist0bar": gh0}
    if s.kind == "hist":
        adcomb.hist_fwd(s.op, s.m, s.keys, s.x, None, s.y, s.saved)
        adcomb.hist_vjp(s.op, s.m, s.keys, s.x, None, s.y, s.saved, s.hb, valsbar=s.xb)
        return {"hist": s.y, "valsbar": s.xb}
    if s.kind == "scan":
        adcomb.scan_fwd(s.op, s.x, s.y)
        adcomb.scan_vjp(s.op, s.x, s.y, s.yb, xbar=s.xb)
        return {"y": s.y, "xbar": s.xb}
    if s.kind == "reduce":
        adcomb.reduce_fwd(s.op, s.x, s.y, s.saved)
        adcomb.reduce_vjp(s.op, s.x, s.y, s.saved, s.yb, xbar=s.xb)
        return {"y": s.y, "xbar": s.xb}
    if s.kind == "rows":
        adcomb.tscan_fwd(s.ops, s.x, s.y)
        adcomb.tscan_vjp(s.ops, s.x, s.y, s.yb, xbar=s.xb)
        return {"y": s.y, "xbar": s.xb}
    if s.kind == "vscan":
        adcomb.vscan_fwd(s.op, s.x, s.y)
        adcomb.vscan_vjp(s.op, s.x, s.y, s.yb, xbar=s.xb)
        return {"y": s.y, "xbar": s.xb}
    p = s.problem
    p.replay_forward()
    p.replay_backward()
    return {"loss": p.loss, "hist": p.hist, "scan": p.scan, "valsbar": p.valsbar}


# ------------------------------------------------- the same in 64 bits -----
def _rev_cumsum(x):
    return torch.flip(torch.cumsum(torch.flip(x, (0,)), 0), (0,))


def _linrec(c, b, reset=None):
    """y_i = b_i + c_i y_{i-1} (y_{-1} = 0) by doubling; a True in ``reset`` starts afresh at i."""
    b, c = b.clone(), c.clone()
    if reset is not None:
        c[reset] = 0
    c[0] = 0
    o, n = 1, b.shape[0]
    while o < n and bool((c != 0).any()):
        nb = b[o:] + (c[o:] if b.dim() == 1 else c[o:, None]) * b[:-o]
        c[o:] = c[o:] * c[:-o]
        b[o:] = nb
        o *= 2
    return b


def _shift(y, first):
    """y_{i-1}, y_{-1} = first."""
    out = torch.empty_like(y)
    out[1:] = y[:-1]
    out[0] = first
    return out


def _next(x, last):
    out = torch.empty_like(x)
    out[:-1] = x[1:]
    out[-1] = last
    return out


def _rev_linrec(c_next, yb):
    """lambda_i = yb_i + c_next_i lambda_{i+1}."""
    return torch.flip(_linrec(torch.flip(c_next, (0,)), torch.flip(yb, (0,))), (0,))


def _mm(a, b):
    """Products of small matrices, [n, q, q] each."""
    q = a.shape[-1]
    out = a[:, :, 0, None] * b[:, None, 0, :]
    for k in range(1, q):
        out += a[:, :, k, None] * b[:, None, k, :]
    return out


def _mat_scan(x, yb):
    n, q = x.shape[0], math.isqrt(x.shape[1])
    m = x.reshape(n, q, q)
    y, o = m.clone(), 1
    while o < n:
        y[o:] = _mm(y[:-o], y[o:])
        o *= 2
    v = torch.flip(yb.reshape(n, q, q), (0,)).clone()  # L_i = Ybar_i + L_{i+1} M_{i+1}^T
    c = torch.zeros_like(v)
    c[1:] = torch.flip(m[1:], (0,)).transpose(1, 2)
    o = 1
    while o < n and bool((c != 0).any()):
        nv = v[o:] + _mm(v[:-o], c[o:])
        nc = torch.zeros_like(c)
        nc[o:] = _mm(c[:-o], c[o:])
        v[o:], c = nv, nc
        o *= 2
    prev = _shift(y, torch.eye(q, dtype=y.dtype, device=y.device))
    return y.reshape(n, -1), _mm(prev.transpose(1, 2), torch.flip(v, (0,))).reshape(n, -1)


def _scan64(op, x, yb):
    if op == "add":
        return torch.cumsum(x, 0), _rev_cumsum(yb)
    if op == "mul":
        y = torch.cumprod(x, 0)
        return y, _shift(y, 1.0) * _rev_linrec(_next(x, 1.0), yb)
    if op == "max":
        y = torch.cummax(x, 0).values
        won = torch.ones(x.shape, dtype=torch.bool, device=x.device)
        won[1:] = y[1:] > y[:-1]
        # lambda at a winner sums ybar up to the next winner: a segmented reverse sum
        tot = _rev_cumsum(yb)
        idx = torch.arange(x.shape[0], device=x.device).reshape(-1, *([1] * (x.dim() - 1))).expand(x.shape)
        nxt = torch.flip(torch.cummin(torch.flip(torch.where(won, idx, x.shape[0]), (0,)), 0).values, (0,))
        after = _next(nxt, x.shape[0])
        pad = torch.cat([tot, torch.zeros_like(tot[:1])], 0)
        return y, torch.where(won, tot - torch.gather(pad, 0, after), torch.zeros_like(tot))
    if op == "lin":
        b, c = x[:, 0], x[:, 1]
        B, C = _linrec(c, b), torch.cumprod(c, 0)
        lam = _rev_linrec(_next(c, 1.0), yb)
        return torch.stack([B, C], 1), torch.stack([lam[:, 0], lam[:, 0] * _shift(B, 0.0) + lam[:, 1] * _shift(C, 1.0)], 1)
    if op == "sop":
        p, t = x[:, 0], x[:, 1]
        S = torch.cumsum(t, 0)
        P = torch.cumsum(p + _shift(S, 0.0) * t, 0)
        lp = _rev_cumsum(yb[:, 0])
        nx = _next(t, 0.0) * _next(lp, 0.0)
        ls = _rev_cumsum(yb[:, 1] + nx)
        return torch.stack([P, S], 1), torch.stack([lp, _shift(S, 0.0) * lp + ls], 1)
    return _mat_scan(x, yb)


def _select64(op, m, keys, v, hb):
    """Best value per bin, and its adjoint at the lowest index that holds it (empty bins: the neutral element)."""
    mx = op == "max"
    best = torch.full((m,), -math.inf if mx else math.inf, dtype=v.dtype, device=v.device)
    best.scatter_reduce_(0, keys, v, "amax" if mx else "amin")
    n = v.shape[0]
    at = torch.arange(n, device=v.device)
    first = torch.full((m,), n, dtype=torch.int64, device=v.device)
    hit = v == best[keys]
    first.scatter_reduce_(0, keys[hit], at[hit], "amin")
    vb = torch.zeros_like(v)
    full = first < n
    vb[first[full]] = hb[full]
    return best, first, vb


def _hist64(op, m, keys, x, hb):
    keys = keys.long()
    if op == "add":
        return torch.zeros(m, dtype=x.dtype, device=x.device).index_add_(0, keys, x), hb[keys]
    if op in ("min", "max"):
        best, _, vb = _select64(op, m, keys, x, hb)
        return best, vb
    if op == "mul":
        zero = x == 0
        n0 = torch.zeros(m, dtype=x.dtype, device=x.device).index_add_(0, keys, zero.to(x.dtype))
        p = torch.ones(m, dtype=x.dtype, device=x.device)
        p.scatter_reduce_(0, keys, torch.where(zero, torch.ones_like(x), x), "prod")
        a = (p * hb)[keys]
        kz = n0[keys]
        one = torch.where(zero & (kz == 1), a, torch.zeros_like(a))
        return torch.where(n0 > 0, torch.zeros_like(p), p), torch.where(kz == 0, a / x, one)
    order = torch.argsort(keys, stable=True)  # lin: segmented recurrences over the values sorted by bin
    k, v = keys[order], x[order]
    start = torch.ones(k.shape, dtype=torch.bool, device=k.device)
    start[1:] = k[1:] != k[:-1]
    end = _next(start, True)
    b, c = v[:, 0], v[:, 1]
    B = _linrec(c, b, start)
    logc = torch.cumsum(torch.log(c), 0)  # c > 0: the segments' products from running sums of logarithms
    seg = torch.cumsum(start.long(), 0) - 1
    base = _shift(logc, 0.0)[start][seg]
    C = torch.exp(logc - base)
    last = logc[end][seg]
    rc = torch.exp(last - logc)
    Bp = torch.where(start, torch.zeros_like(B), _shift(B, 0.0))
    Cp = torch.where(start, torch.ones_like(C), _shift(C, 1.0))
    g = hb[k]
    vb = torch.empty_like(x)
    vb[order] = torch.stack([rc * g[:, 0], rc * (Bp * g[:, 0] + Cp * g[:, 1])], 1)
    hist = torch.zeros((m, 2), dtype=x.dtype, device=x.device)
    hist[:, 1] = 1
    hist[k[end]] = torch.stack([B[end], C[end]], 1)
    return hist, vb


def _reduce64(op, x, yb):
    if op == "add":
        return x.sum().reshape(1), yb.expand(x.shape).clone()
    if op == "max":
        xb = torch.zeros_like(x)
        y = x.max()
        xb[torch.nonzero(x == y)[0, 0]] = yb[0]
        return y.reshape(1), xb
    if op == "mul":
        y = x.prod().reshape(1)
        return y, y / x * yb
    b, c = x[:, 0], x[:, 1]
    B, C = _linrec(c, b), torch.cumprod(c, 0)
    r = _next(torch.flip(torch.cumprod(torch.flip(c, (0,)), 0), (0,)), 1.0)
    return torch.stack([B[-1], C[-1]]), torch.stack([r * yb[0], r * (_shift(B, 0.0) * yb[0] + _shift(C, 1.0) * yb[1])], 1)


def _batched64(case, seed):
    desc, keys, vals, inst = _batched_inputs(case, seed)
    vals = vals.double()
    dev = vals.device
    moff, m = torch.from_numpy(desc["bin_off"].copy()).to(dev), torch.from_numpy(desc["m"].copy()).to(dev)
    is_max = torch.from_numpy(desc["op"] == batched.OPCODE["max"]).to(dev)
    total = int((desc["bin_off"] + desc["m"]).max())
    real = keys >= 0
    b = (moff[inst] + keys)[real]
    v, mx = vals[real], is_max[inst][real]
    hist = torch.zeros(total, dtype=torch.float64, device=dev).index_add_(0, b[~mx], v[~mx])
    best, first, _ = _select64("max", total, b[mx], v[mx], torch.zeros(total, dtype=torch.float64, device=dev))
    won = best > 0  # the zero initial value wins ties
    hist[won] = best[won]
    binst = torch.repeat_interleave(torch.arange(len(m), device=dev), torch.diff(torch.cat([moff, moff.new_tensor([total])])))
    run_ = torch.cumsum(hist, 0)
    scan = run_ - _shift(run_, 0.0)[moff][binst]
    inside = torch.arange(total, device=dev) - moff[binst] < m[binst]
    scan = torch.where(inside, scan, torch.zeros_like(scan))
    vb = torch.zeros_like(vals)
    sel = torch.nonzero(real)[:, 0]
    add_at = sel[~mx]
    vb[add_at] = (m[inst[add_at]] - keys[add_at]).double()
    max_at = sel[mx]
    j = torch.nonzero(won)[:, 0]
    vb[max_at[first[j]]] = (m[binst[j]] - (j - moff[binst[j]])).double()
    return {"loss": scan.sum().reshape(1), "hist": hist, "scan": scan, "valsbar": vb}


def exact(case, seed):
    """What run() returns for these inputs, in 64 bits."""
    if case["kind"] == "batched":
        return _batched64(case, seed)
    s = _inputs(case, seed)
    x = s.x.double()
    if s.kind == "step":
        k = s.keys.long()
        hb, rb, sb = s.hb.double(), s.rb.double(), s.sb.double()
        return {"hist": s.h0.double().index_add(0, k, x), "sum": x.sum(), "scan": torch.cumsum(x, 0),
                "xbar": hb[k] + rb + _rev_cumsum(sb), "hist0bar": hb}
    if s.kind == "hist":
        y, xb = _hist64(s.op, s.m, s.keys, x, s.hb.double())
        return {"hist": y, "valsbar": xb}
    yb = s.yb.double()
    if s.kind == "reduce":
        y, xb = _reduce64(s.op, x, yb)
    elif s.kind == "rows":
        parts = [_scan64(s.op, x[:, 2 * c:2 * c + 2], yb[:, 2 * c:2 * c + 2]) for c in range(len(s.ops))]
        y, xb = torch.cat([p[0] for p in parts], 1), torch.cat([p[1] for p in parts], 1)
    else:
        y, xb = _scan64(s.op, x, yb)
    return {"y": y, "xbar": xb}
