"""What this library's users have it do, as cases that can be timed.

Every case is one whole pass through the public entry points of
``paper_2609_31980_gb300.frnn``: a grid build and the query that follows it
(as every new event needs both), or one of the calls that do the two in one.

Kinds:

* ``self``: build + self-query, dense rows (the plain call).
* ``cross``: build over the references + a query set of its own.
* ``compact``: build + count-first compact rows with full degrees.
* ``host``: page-locked host buffers in and out, compact rows, one call.
* ``batch``: many uneven events in one batched call.
* ``tc``: the self-query through the tensor-core pre-filter (three axes).

Point sets are drawn on the GPU from the seed alone: ``event`` sets are
Gaussian clusters in [-1, 1]^D plus a uniform background (the shape of a
tracking event in its embedding space), ``uniform`` sets fill [0, 1)^D.
Continuous batching over host buffers (``Context.serve``) is not a case of its
own: it paces itself by the clock and runs the batched call.
"""
from __future__ import annotations

import ctypes
import math

import numpy as np
import torch

from paper_2609_31980_gb300 import frnn

DEVICE = "cuda"

# recipes of the tracking-like events by dimension: (radius, cluster sigma)
R8, S8 = 0.1, 0.02      # up to D = 10: most of a cluster lies within r of its points
R12, S12 = 0.12, 0.025  # above: about half of it


def listed():
    return [
        # the smallest call: one small point set, where launches and latency are all there is
        {"name": "uniform_4096x3", "kind": "self", "points": "uniform", "n": 4096, "d": 3,
         "r": 0.05, "k": 32},
        # the smallest event of a serving stream (sizes log-uniform from 20,000), an odd size
        {"name": "event_20011x8", "kind": "self", "points": "event", "n": 20011, "d": 8,
         "r": R8, "k": 64, "per": 30, "sigma": S8},
        # the tracking-like event of the headline benchmark
        {"name": "event_300000x8", "kind": "self", "points": "event", "n": 300000, "d": 8,
         "r": R8, "k": 64, "per": 30, "sigma": S8},
        # the high-dimensional event
        {"name": "event_500000x12", "kind": "self", "points": "event", "n": 500000, "d": 12,
         "r": R12, "k": 128, "per": 25, "sigma": S12},
        # an event of the paper's size, radius and K whose mean degree is the
        # paper's (9,279,672 edges / 271,663 points = 34): compact rows, as
        # rows of K = 1000 are mostly padding
        {"name": "compact_271663x12", "kind": "compact", "points": "event", "n": 271663, "d": 12,
         "r": R12, "k": 1000, "per": 84, "sigma": S12},
        # a large low-dimensional point cloud
        {"name": "uniform_1000000x3", "kind": "self", "points": "uniform", "n": 1000000, "d": 3,
         "r": 0.01, "k": 32},
        # four coordinates, all of them gridded
        {"name": "uniform_300000x4", "kind": "self", "points": "uniform", "n": 300000, "d": 4,
         "r": 0.05, "k": 32},
        # new points looked up in an event's grid: queries that are not the references
        {"name": "cross_300000_100003x8", "kind": "cross", "points": "event", "n": 300000,
         "m": 100003, "d": 8, "r": R8, "k": 64, "per": 30, "sigma": S8},
        # a stream of uneven events taken several at a time
        {"name": "batch_16x8", "kind": "batch", "points": "event", "events": 16, "lo": 50000,
         "hi": 350000, "sizes": 4, "d": 8, "r": R8, "k": 64, "per": 30, "sigma": S8},
        # the headline event from a program whose data lives in host memory
        {"name": "host_300000x8", "kind": "host", "points": "event", "n": 300000, "d": 8,
         "r": R8, "k": 64, "per": 30, "sigma": S8},
        # the high-dimensional event through the tensor-core pre-filter
        {"name": "tc_500000x12", "kind": "tc", "points": "event", "n": 500000, "d": 12,
         "r": R12, "k": 128, "per": 25, "sigma": S12},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _recipe(d):
    return (R8, S8) if d <= 10 else (R12, S12)


def draw(rng):
    kind = rng.choice(["small", "event", "event", "high", "compact", "uniform", "cross", "batch",
                       "host", "tc"])
    if kind in ("small", "uniform"):
        # sizes from a thousand points to the largest cloud, the radius from
        # the mean number of neighbours (2 to 10, as in the listed sets)
        n = _log_int(rng, 1000, 20000) if kind == "small" else _log_int(rng, 20000, 1000000)
        d = rng.choice([2, 3, 3, 4])
        deg = rng.uniform(2.0, 10.0)
        ball = math.pi ** (d / 2) / math.gamma(d / 2 + 1)
        r = round((deg / (n * ball)) ** (1.0 / d), 5)
        return {"kind": "self", "points": "uniform", "n": n, "d": d, "r": r,
                "k": rng.choice([16, 32, 33, 64])}
    if kind == "high":
        d = rng.randint(9, 16)
        n = _log_int(rng, 20000, 500000)
    elif kind == "tc":
        d = rng.randint(10, 16)
        n = _log_int(rng, 50000, 500000)
    elif kind == "compact":
        d = rng.randint(8, 13)
        n = _log_int(rng, 20000, 271663)
    else:
        d = rng.randint(5, 10)
        n = _log_int(rng, 20000, 400000)
    r, sigma = _recipe(d)
    c = {"kind": {"event": "self", "high": "self"}.get(kind, kind), "points": "event", "n": n,
         "d": d, "r": r, "k": rng.choice([32, 50, 64, 100, 128]), "per": rng.randint(15, 30),
         "sigma": sigma}
    if kind == "compact":
        c["per"] = rng.randint(30, 84)
        c["k"] = rng.choice([200, 500, 1000])
    elif kind == "cross":
        c["m"] = _log_int(rng, 5000, n)
    elif kind == "batch":
        del c["n"]
        c["events"] = rng.randint(2, 16)
        c["lo"], c["hi"] = 20000, _log_int(rng, 60000, 300000)
        c["sizes"] = rng.randint(0, 1 << 20)
        c["k"] = rng.choice([32, 50, 64])
    return c


# ---------------------------------------------------------------- inputs


def _points(case, n, seed):
    """[n, d] float32 points of the case's distribution, on the GPU."""
    g = torch.Generator(device=DEVICE).manual_seed(seed)
    d = case["d"]
    if case["points"] == "uniform":
        return torch.rand((n, d), generator=g, device=DEVICE, dtype=torch.float64).float()
    per = case["per"]
    nc = int(round(0.8 * n / per))
    centres = torch.rand((nc, d), generator=g, device=DEVICE, dtype=torch.float64) * 2 - 1
    pts = centres.repeat_interleave(per, dim=0)
    pts += torch.randn(pts.shape, generator=g, device=DEVICE, dtype=torch.float64) * case["sigma"]
    nb = n - nc * per
    if nb > 0:
        bg = torch.rand((nb, d), generator=g, device=DEVICE, dtype=torch.float64) * 2 - 1
        pts = torch.cat([pts, bg])
    order = torch.randperm(pts.shape[0], generator=g, device=DEVICE)[:n]
    return pts[order].float().contiguous()


def _queries(case, refs, seed):
    """m query points: three in four near a reference (as new hits of the
    same tracks are), the rest uniform over the same box."""
    g = torch.Generator(device=DEVICE).manual_seed(seed)
    m, d = case["m"], case["d"]
    near = torch.randint(0, refs.shape[0], (m,), generator=g, device=DEVICE)
    q = refs[near].double()
    q += torch.randn((m, d), generator=g, device=DEVICE, dtype=torch.float64) * case["sigma"]
    far = torch.rand((m, 1), generator=g, device=DEVICE, dtype=torch.float64) < 0.25
    box = torch.rand((m, d), generator=g, device=DEVICE, dtype=torch.float64) * 2 - 1
    return torch.where(far, box, q).float().contiguous()


def _sizes(case):
    g = np.random.Generator(np.random.PCG64(case["sizes"]))
    return [int(x) for x in g.integers(case["lo"], case["hi"] + 1, size=case["events"])]


def _inputs(case, seed):
    """The case's point sets: (refs or list of events, queries or None)."""
    if case["kind"] == "batch":
        return [_points(case, n, seed * 1000003 + e) for e, n in enumerate(_sizes(case))], None
    refs = _points(case, case["n"], seed * 1000003)
    return refs, (_queries(case, refs, seed * 1000003 + 1) if case["kind"] == "cross" else None)


def _expected_edges(case, n, m):
    """Expected pairs of m queries among n references: in-cluster pairs
    (their distance is sigma sqrt(2 chi2_d)) plus an even spread."""
    d, r = case["d"], case["r"]
    ball = math.pi ** (d / 2) / math.gamma(d / 2 + 1) * r ** d
    if case["points"] == "uniform":
        return m * n * ball
    p = float(torch.special.gammainc(torch.tensor(d / 2.0, dtype=torch.float64),
                                     torch.tensor(r * r / (4 * case["sigma"] ** 2), dtype=torch.float64)))
    return m * (0.8 * (case["per"] - 1) * p + n * ball / 2 ** d)


def _edge_capacity(case):
    """Entries a compact output is given: twice the expected pairs, which the
    spread of the degrees does not come near."""
    n = case["n"]
    return int(2 * _expected_edges(case, n, n)) + 64 * 1024


def _dense_out(m, k):
    return (torch.empty(m, dtype=torch.int32, device=DEVICE),
            torch.empty((m, k), dtype=torch.int32, device=DEVICE),
            torch.empty((m, k), dtype=torch.float32, device=DEVICE))


def _pinned(shape, dtype):
    return torch.zeros(shape, dtype=dtype).pin_memory().numpy()


def prepare(case, seed):
    refs, queries = _inputs(case, seed)
    ctx = frnn.Context()
    s = {"case": case, "ctx": ctx, "refs": refs, "queries": queries}
    kind, k = case["kind"], case["k"]
    if kind == "host":
        pts = _pinned(tuple(refs.shape), torch.float32)
        pts[...] = refs.cpu().numpy()
        cap = _edge_capacity(case)
        s["refs"] = pts
        s["out"] = (_pinned((case["n"] + 1,), torch.int64), _pinned((cap,), torch.int32),
                    _pinned((cap,), torch.float32))
        return s
    if kind == "batch":
        s["out"] = [_dense_out(p.shape[0], k) for p in refs]
        return s
    if kind == "tc":
        ctx.set_option(frnn.FRNN_OPT_GRID_NAXES, 3)
    # the grid is kept from event to event and rebuilt in place
    s["grid"] = ctx.build_grid(refs, case["r"])
    if kind == "compact":
        n, cap = case["n"], _edge_capacity(case)
        s["offsets"] = torch.zeros(n + 1, dtype=torch.int64, device=DEVICE)
        s["degree"] = torch.zeros(n, dtype=torch.int32, device=DEVICE)
        s["idx"] = torch.zeros(cap, dtype=torch.int32, device=DEVICE)
        s["dist2"] = torch.zeros(cap, dtype=torch.float32, device=DEVICE)
    else:
        s["out"] = _dense_out(case["m"] if kind == "cross" else case["n"], k)
    return s


# ---------------------------------------------------------------- one pass


def _check(ctx, status):
    if status != frnn.FRNN_OK:
        raise frnn.FrnnError(status, frnn.frnn_last_error(ctx.handle).decode())


def run(state):
    case, ctx = state["case"], state["ctx"]
    kind, r, k = case["kind"], case["r"], case["k"]
    if kind == "host":
        ctx.self_query_host_csr(state["refs"], r, k, out=state["out"])
        return state["out"]
    if kind == "batch":
        return ctx.query_batched(state["refs"], r, k, outs=state["out"])
    refs = state["refs"]
    grid = ctx.build_grid(refs, r, grid=state["grid"])
    if kind == "cross":
        return ctx.query(grid, state["queries"], r, k, self_query=False, out=state["out"])
    if kind == "tc":
        return ctx.query(grid, refs, r, k, path="tc", out=state["out"])
    if kind == "compact":
        # count pass, then the rows into a buffer the caller keeps
        n_edges = ctypes.c_int64(0)
        ptr = lambda t: ctypes.c_void_p(t.data_ptr())  # noqa: E731
        _check(ctx, frnn.frnn_query_csr_count(
            ctx.handle, grid.handle, ptr(refs), refs.shape[0], r, k, frnn.FRNN_SELF_QUERY,
            ptr(state["offsets"]), ptr(state["degree"]), ctypes.byref(n_edges)))
        if n_edges.value > state["idx"].numel():
            raise RuntimeError("more edges than the caller's buffer holds")
        _check(ctx, frnn.frnn_query_csr_fill(ctx.handle, ptr(state["idx"]), ptr(state["dist2"])))
        return state["offsets"], state["idx"], state["dist2"], state["degree"]
    return ctx.query(grid, refs, r, k, out=state["out"])


# ---------------------------------------------------------------- work


def work(case):
    """Inputs read once, outputs written once; the squared distances of the
    pairs that are returned (3 D operations each)."""
    d, k, kind = case["d"], case["k"], case["kind"]
    sizes = _sizes(case) if kind == "batch" else [case["n"]]
    nbytes = flops = 0.0
    for n in sizes:
        m = case.get("m", n)
        edges = _expected_edges(case, n, m)
        nbytes += 4.0 * d * (n + (m if kind == "cross" else 0))
        if kind == "compact":
            nbytes += 8.0 * (m + 1) + 4.0 * m + 8.0 * edges
        elif kind == "host":
            nbytes += 8.0 * (m + 1) + 8.0 * edges
        else:
            nbytes += 4.0 * m + 8.0 * m * k
        flops += 3.0 * d * edges
    return {"bytes": nbytes, "flops": flops}


# ---------------------------------------------------------------- 64 bits


def _pairs(refs, queries, r, self_query):
    """(query, squared distance) of every pair within r in float64, ordered by
    query, distance and reference: windows of the points sorted along the
    last coordinate."""
    x = refs.double()
    q = x if self_query else queries.double()
    r2 = float(np.float32(r)) ** 2
    reach = float(np.float32(r)) * (1 + 1e-6)
    xo = torch.argsort(x[:, -1])
    qo = torch.argsort(q[:, -1])
    xs, qs = x[xo], q[qo]
    key = xs[:, -1].contiguous()
    step = 2048
    first = torch.arange(0, qs.shape[0], step, device=x.device)
    last = torch.clamp(first + step, max=qs.shape[0]) - 1
    lo = torch.searchsorted(key, qs[first, -1] - reach).tolist()
    hi = torch.searchsorted(key, qs[last, -1] + reach, right=True).tolist()
    got = []
    for c, (a, b) in enumerate(zip(lo, hi)):
        part = qs[c * step:(c + 1) * step]
        win = xs[a:b]
        d2 = torch.zeros((part.shape[0], win.shape[0]), dtype=torch.float64, device=x.device)
        for j in range(x.shape[1]):
            t = part[:, j, None] - win[None, :, j]
            d2.addcmul_(t, t)
        i, j = (d2 <= r2).nonzero(as_tuple=True)
        qi, xj = qo[c * step + i], xo[a + j]
        v = d2[i, j]
        if self_query:
            keep = qi != xj
            qi, xj, v = qi[keep], xj[keep], v[keep]
        got.append((qi, xj, v))
    qi, xj, v = (torch.cat(t) for t in zip(*got))
    for by in (lambda: xj, lambda: v, lambda: qi):   # least significant key first
        o = torch.argsort(by(), stable=True)
        qi, xj, v = qi[o], xj[o], v[o]
    return qi, v


def _truncate(qi, v, m, k):
    """Position of each pair in its query's row, for the pairs kept."""
    counts = torch.bincount(qi, minlength=m)
    start = torch.cumsum(counts, 0) - counts
    pos = torch.arange(qi.shape[0], device=qi.device) - start[qi]
    keep = pos < k
    return qi[keep], pos[keep], v[keep]


def _exact_dense(refs, queries, r, k, self_query):
    m = refs.shape[0] if self_query else queries.shape[0]
    qi, v = _pairs(refs, queries, r, self_query)
    qi, pos, v = _truncate(qi, v, m, k)
    out = torch.full((m, k), math.inf, dtype=torch.float64, device=refs.device)
    out[qi, pos] = v
    return out


def exact(case, seed):
    kind, r, k = case["kind"], case["r"], case["k"]
    refs, queries = _inputs(case, seed)
    if kind == "batch":
        return [(None, None, _exact_dense(p, None, r, k, True)) for p in refs]
    if kind in ("compact", "host"):
        qi, v = _pairs(refs, None, r, True)
        _, _, v = _truncate(qi, v, case["n"], k)
        rows = torch.zeros(_edge_capacity(case), dtype=torch.float64, device=refs.device)
        rows[:v.shape[0]] = v
        if kind == "host":
            return None, None, rows.cpu().numpy()
        return None, None, rows, None
    return None, None, _exact_dense(refs, queries, r, k, kind != "cross")
