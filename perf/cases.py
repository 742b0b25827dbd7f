"""What a user of the library has it do, as cases that can be timed.

A case is one call (or one captured run) of a public entry point of
``paper_2305_16751_gb300.domagg`` on inputs drawn like the workloads of
``workloads.py``, with the sizes of the tests, the benchmark's workloads and
ragged sizes between them:

  forward   domagg.forward on device tensors
  grad      domagg.dominance_sum and its gradient (the autograd step)
  host      domagg.forward_host on pinned host tensors (copies included)
  batch     domagg.domagg_batch: independent problems in one call
  plan      domagg.domagg_plan_run replayed from a CUDA graph

``exact`` computes the definition in 64 bits with torch's own sorts and
cumulative sums and uses nothing of this repository.
"""
import ctypes
import math

import numpy as np
import torch

from paper_2305_16751_gb300 import domagg

DEV = "cuda"


def listed():
    f = "forward"
    return [
        # the smallest problem in use: the first benchmark configuration
        # (integer coordinates, 8-byte weights), called one at a time
        dict(name="m2_small_i64sum", kind=f, m=2, nD=4096, nQ=4096, coords="i32_20", op="sum", wt="i64", nonstrict=0),
        # a small autograd step in three dimensions, ragged sizes
        dict(name="m3_small_grad", kind="grad", m=3, nD=7001, nQ=9003, coords="f32_grid", op="sum", wt="f32",
             nonstrict=0),
        # an ordinary call: a sample of some 10^5 points, ties, odd sizes
        dict(name="m2_mid_f32sum", kind=f, m=2, nD=100003, nQ=65537, coords="f32_tied", op="sum", wt="f32",
             nonstrict=0),
        # end to end from host memory: the maximum of int32 weights, fewer
        # queries than data
        dict(name="m2_host_i32max", kind="host", m=2, nD=2**22, nQ=1500001, coords="f32_tied", op="max", wt="i32",
             nonstrict=0),
        # the headline: 2^24 points per side, a quarter of them tied
        dict(name="m2_large_f32sum", kind=f, m=2, nD=2**24, nQ=2**24, coords="f32_tied", op="sum", wt="f32",
             nonstrict=0),
        # the training step: forward and backward at 2^22 per side
        dict(name="m2_grad", kind="grad", m=2, nD=2**22, nQ=2**22, coords="f32_grid", op="sum", wt="f32",
             nonstrict=0),
        # three dimensions, clustered integer coordinates, 8-byte weights
        dict(name="m3_gmm_i64sum", kind=f, m=3, nD=2**21, nQ=2**21, coords="i32_gmm", op="sum", wt="i64",
             nonstrict=0),
        # the empirical CDF of one sample at both samples' points: counts
        # with every coordinate compared non-strictly
        dict(name="m3_ecdf_count", kind=f, m=3, nD=300007, nQ=600011, coords="f32_ecdf", op="count", wt="i64",
             nonstrict=7),
        # one dimension: prefix sums at the rank of every query
        dict(name="m1_prefix_f32sum", kind=f, m=1, nD=2**22, nQ=2**21 + 12345, coords="f32_grid", op="sum", wt="f32",
             nonstrict=0),
        # four dimensions, the minimum of float weights
        dict(name="m4_f32min", kind=f, m=4, nD=12000, nQ=9001, coords="i32_31", op="min", wt="f32", nonstrict=0),
        # independent problems of two and three dimensions, sizes spread
        # over [256, 2^18] (the batch workload's recipe), one call
        dict(name="batch_mixed", kind="batch", k=256, lo=256, hi=2**18, coords="i32_31", op="sum", wt="f32",
             nonstrict=0),
        # a planned batch of small problems replayed from a CUDA graph, as a
        # server runs it
        dict(name="plan_small", kind="plan", k=192, lo=256, hi=4096, coords="i32_31", op="sum", wt="f32",
             nonstrict=0),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the listed ranges: sizes log-uniform and mostly odd,
    any supported operator with its weights."""
    kind = rng.choice(["forward", "forward", "forward", "grad", "host", "batch", "plan"])
    if kind in ("batch", "plan"):
        hi = _log(rng, 2**15, 2**18) if kind == "batch" else _log(rng, 2**10, 2**13)
        return dict(kind=kind, k=rng.randint(24, 256 if kind == "batch" else 320), lo=256, hi=hi,
                    coords=rng.choice(["i32_31", "i32_20", "f32_grid"]), op="sum", wt=rng.choice(["f32", "i64"]),
                    nonstrict=0)
    m = rng.choice([1, 2, 2, 2, 3, 3, 4]) if kind == "forward" else rng.choice([2, 2, 3])
    top = {1: 2**23, 2: 2**23, 3: 2**20, 4: 12000}[m]
    nD = _log(rng, 1000, top)
    nQ = min(top, max(500, int(nD * math.exp(rng.uniform(-1.2, 1.2)))))
    op, wt = rng.choice([("sum", "f32"), ("sum", "f32"), ("sum", "i64"), ("count", "i64"), ("max", "i32"),
                         ("min", "f32")])
    nonstrict = 0
    if kind == "grad":
        op, wt = "sum", "f32"
    if kind == "forward" and rng.random() < 0.25:
        nonstrict = rng.randrange(1, 1 << m)
    return dict(kind=kind, m=m, nD=nD, nQ=nQ,
                coords=rng.choice(["f32_tied", "f32_grid", "i32_20", "i32_31", "i32_gmm", "f32_ecdf"]), op=op, wt=wt,
                nonstrict=nonstrict)


# --- inputs -------------------------------------------------------------------

def _points(n, m, coords, g, shift=0.0):
    """n points of dimension m: the coordinate distributions of workloads.py."""
    if coords in ("f32_grid", "f32_tied"):  # [0, 1) on the 2^-24 grid; "tied": a quarter of the points on 2^-16
        x = torch.randint(0, 1 << 24, (n, m), device=DEV, generator=g, dtype=torch.int32)
        if coords == "f32_tied":
            q = torch.rand((n, 1), device=DEV, generator=g) < 0.25
            x = torch.where(q, x & ~0xff, x)
        return x.to(torch.float32) * 2.0**-24
    if coords == "i32_20":
        return torch.randint(0, 1 << 20, (n, m), device=DEV, generator=g, dtype=torch.int32)
    if coords == "i32_31":
        return torch.randint(0, (1 << 31) - 1, (n, m), device=DEV, generator=g, dtype=torch.int32)
    if coords == "f32_ecdf":  # N(shift, 1) on a 2^-8 grid
        return torch.round((torch.randn((n, m), device=DEV, generator=g) + shift) * 256.0) / 256.0
    assert coords == "i32_gmm"  # 16 Gaussian components, clipped to [0, 2^24)
    gm = torch.Generator(device=DEV).manual_seed(g.initial_seed() % 1000 + 77)  # the same mixture for D and Q
    mean = torch.rand((16, m), device=DEV, generator=gm) * 2.0**24
    sig = 2.0**16 + torch.rand((16, m), device=DEV, generator=gm) * (2.0**20 - 2.0**16)
    c = torch.randint(0, 16, (n,), device=DEV, generator=g)
    x = torch.randn((n, m), device=DEV, generator=g) * sig[c] + mean[c]
    return torch.round(x).clamp(0, 2**24 - 1).to(torch.int32)


def _weights(n, wt, g):
    if wt == "f32":
        return torch.randn(n, device=DEV, generator=g)
    if wt == "i64":
        return torch.randint(-1000, 1001, (n,), device=DEV, generator=g)
    return torch.randint(-2**30, 2**30, (n,), device=DEV, generator=g).to(torch.int32)


def _problem(case, seed):
    """D, Q, w (and the loss coefficients of a gradient case)."""
    g = torch.Generator(device=DEV).manual_seed(int(seed))
    D = _points(case["nD"], case["m"], case["coords"], g)
    Q = _points(case["nQ"], case["m"], case["coords"], g, 0.05)
    w = _weights(case["nD"], case["wt"], g)
    c = torch.randn(case["nQ"], device=DEV, generator=g)
    return D, Q, w, c


def _batch_shapes(case):
    """Per instance m (2 or 3) and points per side, log-uniform in [lo, hi]:
    the same for every seed, as a server's batch slots are."""
    r = np.random.default_rng(case["k"] * 1000003 + case["hi"])
    ms = r.integers(2, 4, size=case["k"])
    n = np.exp(r.uniform(math.log(case["lo"]), math.log(case["hi"]), size=case["k"])).astype(np.int64)
    n = np.clip(n, case["lo"], case["hi"])
    # the largest size and both dimensions are always there
    n[0], ms[0], ms[1] = case["hi"], 3, 2
    return [int(x) for x in ms], [int(x) for x in n]


def _batch(case, seed):
    """Every instance's D, Q, w as consecutive rows of shared buffers."""
    g = torch.Generator(device=DEV).manual_seed(int(seed))
    ms, ns = _batch_shapes(case)
    total = sum(m * n for m, n in zip(ms, ns))
    Dall = _points(total, 1, case["coords"], g).reshape(-1)
    Qall = _points(total, 1, case["coords"], g).reshape(-1)
    wall = _weights(sum(ns), case["wt"], g)
    return ms, ns, Dall, Qall, wall


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("forward", "grad", "host"):
        D, Q, w, c = _problem(case, seed)
        w = None if case["op"] == "count" else w
        if kind == "grad":
            w.requires_grad_(True)
        if kind == "host":  # a user's host arrays, in pinned memory
            D, Q = D.cpu().pin_memory(), Q.cpu().pin_memory()
            w = None if w is None else w.cpu().pin_memory()
        return dict(kind=kind, op=case["op"], nonstrict=case["nonstrict"], D=D, Q=Q, w=w, c=c)
    ms, ns, Dall, Qall, wall = _batch(case, seed)
    out = torch.empty_like(wall)
    arr = (domagg.domagg_instance * len(ns))()
    pc, pn = 0, 0
    for i, (m, n) in enumerate(zip(ms, ns)):
        arr[i] = domagg.domagg_instance(m, n, n, Dall[pc:].data_ptr(), Qall[pc:].data_ptr(), wall[pn:].data_ptr(),
                                        out[pn:].data_ptr())
        pc += m * n
        pn += n
    types = (domagg.DTYPES["f32" if case["coords"].startswith("f32") else "i32"], domagg.DTYPES[case["wt"]],
             domagg.OPS[case["op"]])
    state = dict(kind=kind, arr=arr, types=types, out=out, keep=(Dall, Qall, wall))
    if kind == "plan":
        state["plan"] = _Plan(arr, types)
    return state


class _Plan:
    """A planned batch and the CUDA graph that replays it (released together)."""

    def __init__(self, arr, types):
        side = torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        s = ctypes.c_void_p(side.cuda_stream)
        self.p = domagg.domagg_batch_plan(0, len(arr), arr, *types, 0.25, s)
        self.graph = torch.cuda.CUDAGraph()
        with torch.cuda.stream(side):
            with torch.cuda.graph(self.graph, stream=side):
                domagg.domagg_plan_run(self.p, s)
        torch.cuda.current_stream().wait_stream(side)

    def __del__(self):
        if getattr(self, "p", None):
            torch.cuda.synchronize()
            self.graph = None
            domagg.domagg_plan_destroy(self.p)
            self.p = None


def run(state):
    kind = state["kind"]
    if kind == "forward":
        return domagg.forward(state["D"], state["Q"], state["w"], state["op"], nonstrict=state["nonstrict"])
    if kind == "host":
        return domagg.forward_host(state["D"], state["Q"], state["w"], state["op"])
    if kind == "grad":
        out = domagg.dominance_sum(state["D"], state["Q"], state["w"])
        (gw,) = torch.autograd.grad(out, state["w"], state["c"])
        return out.detach(), gw
    if kind == "batch":
        s = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
        domagg.domagg_batch(domagg.handle(0), len(state["arr"]), state["arr"], *state["types"], s)
    else:
        state["plan"].graph.replay()
    return state["out"]


def work(case):
    """Inputs read once and outputs written once.  Per F application of the
    range-tree decomposition one operation: half of the levels of each of
    the m-1 ranks, per point."""
    wb = {"f32": 4, "i32": 4, "i64": 8}[case["wt"]]
    if case["kind"] in ("batch", "plan"):
        ms, ns = _batch_shapes(case)
        probs = [(m, n, n) for m, n in zip(ms, ns)]
    else:
        probs = [(case["m"], case["nD"], case["nQ"])]
    nbytes = flops = 0.0
    for m, nD, nQ in probs:
        wr = 0 if case["op"] == "count" else wb
        b = nD * (4 * m + wr) + nQ * (4 * m + wb)
        f = (nD + nQ) * (math.log2(nD + nQ) / 2) ** (m - 1)
        if case["kind"] == "grad":  # and back: grad_out read, grad_w written
            b, f = 2 * b, 2 * f
        nbytes += b
        flops += f
    return {"bytes": nbytes, "flops": flops}


# --- the definition in 64 bits ------------------------------------------------

def _order(Dc, Qc, strict, group):
    """Positions of data and queries in one total order (per group) in which
    d before q says d < q (strict) or d <= q."""
    x = torch.cat([Dc, Qc])
    nD = Dc.shape[0]
    _, x = torch.unique(x, return_inverse=True)
    isq = torch.zeros_like(x)
    isq[nD:] = 1
    key = (group * (x.max() + 1) + x) * 2 + ((1 - isq) if strict else isq)
    pos = torch.empty_like(key)
    pos[torch.argsort(key, stable=True)] = torch.arange(key.numel(), device=key.device)
    return pos


def _scan(vals, seg, op):
    """Per position, F over the earlier values of its segment (segments are
    consecutive)."""
    if op == "sum":
        inc = torch.cumsum(vals, 0)
        exc = inc - vals
        head = torch.ones_like(seg, dtype=torch.bool)
        head[1:] = seg[1:] != seg[:-1]
        start = torch.cummax(torch.where(head, torch.arange(seg.numel(), device=seg.device), 0), 0).values
        return exc - exc[start]
    # max of non-negative int64 values below 2^32, 0 the unit: a segment's
    # values are lifted above every earlier segment's
    lift = torch.unique_consecutive(seg, return_inverse=True)[1] << 32
    inc = torch.cummax(vals + lift, 0).values
    exc = torch.cat([inc[:1] * 0, inc[:-1]])
    return (exc - lift).clamp_min(0)


def _aggregate(ranks, items, seg, isq, vals, out, op):
    """items: indices in the order (seg, last coordinate); ranks: the
    remaining coordinates' total orders."""
    if not ranks:
        r = _scan(vals[items], seg, op)  # (a query's value is the unit)
        q = isq[items] == 1
        if op == "sum":
            out[items[q]] += r[q]
        else:
            out[items[q]] = torch.maximum(out[items[q]], r[q])
        return
    n = isq.numel()
    bits = max(1, (n - 1).bit_length())
    for lv in range(bits):
        r = ranks[0][items]
        keep = ((r >> lv) & 1) == isq[items]
        sub = items[keep]
        if sub.numel() == 0:
            continue
        s = (seg[keep] << (bits - lv)) | (r[keep] >> (lv + 1))
        s, o = torch.sort(s, stable=True)
        s = torch.unique_consecutive(s, return_inverse=True)[1]
        _aggregate(ranks[1:], sub[o], s, isq, vals, out, op)


def _exact(D, Q, w, op, nonstrict, gD=None, gQ=None):
    """out per query, from the definition (groups gD, gQ: independent problems)."""
    nD, nQ, m = D.shape[0], Q.shape[0], D.shape[1]
    dev = D.device
    gD = torch.zeros(nD, dtype=torch.int64, device=dev) if gD is None else gD
    gQ = torch.zeros(nQ, dtype=torch.int64, device=dev) if gQ is None else gQ
    group = torch.cat([gD, gQ])
    isq = torch.zeros(nD + nQ, dtype=torch.int64, device=dev)
    isq[nD:] = 1
    ranks = [_order(D[:, i].contiguous(), Q[:, i].contiguous(), not (nonstrict >> i) & 1, group) for i in range(m)]
    if op == "count":
        op, w = "sum", torch.ones(nD, dtype=torch.int64, device=dev)
    levels = None
    if op in ("max", "min"):  # by the weights' ranks, 1 up; 0 is the unit
        levels, w = torch.unique(w, return_inverse=True)
        w = (levels.numel() - w) if op == "min" else w + 1
    v = w.to(torch.float64 if w.dtype.is_floating_point else torch.int64)
    vals = torch.cat([v, torch.zeros(nQ, dtype=v.dtype, device=dev)])
    out = torch.zeros_like(vals)
    items = torch.argsort(ranks[-1])
    _aggregate(ranks[:-1], items, group[items], isq, vals, out, "sum" if op == "sum" else "max")
    out = out[nD:]
    if levels is None:
        return out
    if levels.dtype.is_floating_point:
        unit = torch.tensor([-math.inf if op == "max" else math.inf], device=dev, dtype=torch.float64)
        levels = levels.to(torch.float64)
    else:
        unit = torch.tensor([-2**31 if op == "max" else 2**31 - 1], device=dev, dtype=levels.dtype)
    if op == "min":
        levels = levels.flip(0)
    return torch.cat([unit, levels])[out]


def exact(case, seed):
    kind = case["kind"]
    if kind in ("batch", "plan"):
        ms, ns, Dall, Qall, wall = _batch(case, seed)
        dt = torch.float64 if case["wt"] == "f32" else wall.dtype
        out = torch.empty(wall.shape, dtype=dt, device=DEV)
        for m in (2, 3):
            Ds, Qs, rows, grp = [], [], [], []
            pc = pn = 0
            for i, (mi, n) in enumerate(zip(ms, ns)):
                if mi == m:
                    Ds.append(Dall[pc:pc + m * n].reshape(n, m))
                    Qs.append(Qall[pc:pc + m * n].reshape(n, m))
                    rows.append(torch.arange(pn, pn + n, device=DEV))
                    grp.append(torch.full((n,), i, dtype=torch.int64, device=DEV))
                pc += mi * n
                pn += n
            rows, grp = torch.cat(rows), torch.cat(grp)
            out[rows] = _exact(torch.cat(Ds), torch.cat(Qs), wall[rows], case["op"], 0, grp, grp)
        return out
    D, Q, w, c = _problem(case, seed)
    out = _exact(D, Q, w, case["op"], case["nonstrict"])
    if kind == "host":
        return out.cpu()
    if kind == "grad":  # the transposed sum: roles swapped, every order reversed
        neg = (lambda x: -x.to(torch.float64)) if D.dtype == torch.float32 else (lambda x: -x.to(torch.int64))
        return out, _exact(neg(Q), neg(D), c, "sum", 0)
    return out
