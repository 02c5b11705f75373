"""The scan of the automatic grids of up to four dimensions (query_low.cu)
against the oracle bit for bit, at the sizes where it can go wrong: every number
of lanes per query (8 below 12,000 points, 4, 2, 1), remainders of a warp, every
sort width and rows past the list, both row writers, outputs off a 16-byte
boundary, wider neighbourhoods (m = 2, 3), ties, empty neighbourhoods, cross
sets and batches whose warps straddle events."""
import numpy as np
import pytest

from oracle import oracle
from paper_2609_31980_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_2609_31980_gb300 import frnn
    c = frnn.Context()
    yield c
    c.close()


def _same(got, want):
    c, i, d = (t.cpu().numpy() for t in got)
    np.testing.assert_array_equal(c, want[0])
    np.testing.assert_array_equal(i, want[1])
    np.testing.assert_array_equal(d.view(np.uint32), want[2].view(np.uint32))


def _t(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a, np.float32)).cuda()


def _radius(n, D, deg):
    ball = {1: 2.0, 2: np.pi, 3: 4 * np.pi / 3, 4: np.pi ** 2 / 2}[D]
    return float((deg / (n * ball)) ** (1.0 / D))


def _points(n, D, seed):
    """Uniform points, a denser blob, repeated points and a lattice."""
    g = np.random.default_rng(seed)
    p = g.random((n, D), dtype=np.float32)
    k = n // 8
    p[:k] = p[:k] * np.float32(0.25) + np.float32(0.5)
    p[k:2 * k] = np.round(p[k:2 * k] * 16) / 16
    p[2 * k:2 * k + k // 2] = p[: k // 2]
    return p


@pytest.mark.parametrize("D", [1, 2, 3, 4])
@pytest.mark.parametrize("n", [1, 2, 31, 33, 3001, 13001, 25003, 50001])
def test_sizes(ctx, D, n):
    import torch
    p = _points(n, D, 900 + D)
    rows = np.arange(n) if n < 4000 else np.arange(0, n, 17)
    for deg in (3.0, 14.0):
        r = _radius(max(n, 64), D, deg)
        got = ctx.self_query(_t(p), r, 32, path="grid")
        ctx.sync()
        at = torch.from_numpy(rows).cuda()
        _same(tuple(x[at] for x in got), oracle.self_query(p, r, 32, rows=rows))


@pytest.mark.parametrize("K", [1, 3, 4, 8, 20, 31, 44, 64, 68, 128, 200])
@pytest.mark.parametrize("D", [2, 3])
def test_row_widths_and_alignment(ctx, K, D):
    import torch
    n = 5000
    p = _points(n, D, 920)
    r = _radius(n, D, 8.0)
    want = oracle.self_query(p, r, K)
    t = _t(p)
    for off in (0, 1):
        c = torch.empty(n, dtype=torch.int32, device="cuda")
        i = torch.empty(n * K + 4, dtype=torch.int32, device="cuda")[off:off + n * K].view(n, K)
        d = torch.empty(n * K + 4, dtype=torch.float32, device="cuda")[off:off + n * K].view(n, K)
        _same(ctx.self_query(t, r, K, path="grid", out=(c, i, d)), want)
    g = ctx.build_grid(t, r)
    off, ci, cd, deg = ctx.query_csr(g, t, r, K, degree=True)
    ctx.sync()
    keep = np.arange(K)[None, :] < want[0][:, None]
    np.testing.assert_array_equal(np.diff(off.cpu().numpy()), want[0])
    np.testing.assert_array_equal(ci.cpu().numpy(), want[1][keep])
    np.testing.assert_array_equal(cd.cpu().numpy().view(np.uint32), want[2][keep].view(np.uint32))
    np.testing.assert_array_equal(deg.cpu().numpy(), want[3])


@pytest.mark.parametrize("D", [1, 2, 3, 4])
@pytest.mark.parametrize("m", [1, 2, 3])
def test_wider_neighbourhoods_and_cross_sets(ctx, D, m):
    from paper_2609_31980_gb300 import frnn
    p = _points(6000, D, 930 + D)
    q = np.random.default_rng(931).uniform(-0.5, 1.5, size=(777, D)).astype(np.float32)
    r = _radius(6000, D, 6.0)
    ctx.set_option(frnn.FRNN_OPT_CELL_MULT, m)
    try:
        g = ctx.build_grid(_t(p), r)
        got = ctx.query(g, _t(q), r, 24, self_query=False, path="grid")
        ctx.sync()
        _same(got, oracle.frnn(q, p, r, 24))
    finally:
        ctx.set_option(frnn.FRNN_OPT_CELL_MULT, 0)


@pytest.mark.parametrize("sizes", [(5, 0, 17, 300, 1, 2500), (20000, 33, 40001)])
def test_batches(ctx, sizes):
    ev = [_points(max(n, 1), 3, 940 + n)[:n] for n in sizes]
    outs = ctx.query_batched([_t(p.reshape(-1, 3)) for p in ev], 0.04, 32, path="grid")
    ctx.sync()
    for p, o in zip(ev, outs):
        if len(p):
            rows = np.arange(0, len(p), max(1, len(p) // 1000))
            import torch
            at = torch.from_numpy(rows).cuda()
            _same(tuple(x[at] for x in o), oracle.self_query(p, 0.04, 32, rows=rows))
