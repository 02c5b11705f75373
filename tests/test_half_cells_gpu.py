"""The half-cell scan (query_half.cu: the automatic grids from D = 5 on) against
the oracle bit for bit, at the sizes where it can go wrong: chunks of 16, 8 and
4 queries and their remainders, every row width class (16-byte and 4-byte
stores, rows cut below the list, rows past it), outputs that are not 16-byte
aligned, cells on the grid's edges, ties, and queries that are not the
references."""
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


def _points(n, D, seed):
    """Clusters (rows of a few to more than 32 neighbours), background,
    repeated points and points on a lattice of the radius."""
    g = np.random.default_rng(seed)
    a = synth.clustered(max(n // 60, 1), 40, n - n // 3, D, 0.025, seed=(seed, 1))[: n - n // 4]
    b = (g.integers(-2, 3, size=(n - len(a), D)) * 0.125).astype(np.float32)
    p = np.concatenate([a, b])[:n]
    p[n // 2: n // 2 + n // 16] = p[: n // 16]
    return np.ascontiguousarray(p[g.permutation(n)])


@pytest.mark.parametrize("D", [5, 6, 8, 9, 12, 13, 16])
@pytest.mark.parametrize("n", [1, 3, 4, 5, 16, 17, 33, 2500])
def test_small_sets(ctx, D, n):
    import torch
    p = _points(n, D, 800 + D) if n > 33 else synth.uniform(n, D, seed=800 + n, hi=0.2)
    if D >= 9:   # sets this small keep four axes by default: add far points
        p = np.concatenate([p, synth.uniform(16500, D, seed=801, lo=30.0, hi=31.0)])
    t = torch.from_numpy(p).cuda()
    rows = np.arange(min(n, 2500))
    for K in (3, 32, 64):
        got = ctx.self_query(t, 0.125, K, path="grid")
        ctx.sync()
        _same(tuple(x[:len(rows)] for x in got), oracle.self_query(p, 0.125, K, rows=rows))


@pytest.mark.parametrize("K", [1, 2, 4, 5, 16, 31, 36, 100, 128, 200])
def test_row_widths_and_alignment(ctx, K):
    import torch
    p = _points(6000, 8, 820)
    t = torch.from_numpy(p).cuda()
    want = oracle.self_query(p, 0.1, K)
    for off in (0, 1):   # the second: rows that start off a 16-byte boundary
        c = torch.empty(len(p), dtype=torch.int32, device="cuda")
        i = torch.empty(len(p) * K + 4, dtype=torch.int32, device="cuda")[off:off + len(p) * K].view(len(p), K)
        d = torch.empty(len(p) * K + 4, dtype=torch.float32, device="cuda")[off:off + len(p) * K].view(len(p), K)
        _same(ctx.self_query(t, 0.1, K, path="grid", out=(c, i, d)), want)
    g = ctx.build_grid(t, 0.1)
    off, ci, cd, deg = ctx.query_csr(g, t, 0.1, K, degree=True)
    ctx.sync()
    keep = np.arange(K)[None, :] < want[0][:, None]
    np.testing.assert_array_equal(np.diff(off.cpu().numpy()), want[0])
    np.testing.assert_array_equal(ci.cpu().numpy(), want[1][keep])
    np.testing.assert_array_equal(cd.cpu().numpy().view(np.uint32), want[2][keep].view(np.uint32))
    np.testing.assert_array_equal(deg.cpu().numpy(), want[3])


@pytest.mark.parametrize("D", [5, 8, 12])
@pytest.mark.parametrize("axes", [0, 1])
def test_cross_sets_and_axis_choice(ctx, D, axes):
    import torch
    from paper_2609_31980_gb300 import frnn
    refs = np.concatenate([_points(4000, D, 830), synth.uniform(14000, D, seed=831, lo=-1.2, hi=1.2)])
    refs[:, D // 2] *= 3.0   # the widest axes are not the last ones
    q = np.concatenate([_points(1001, D, 832), synth.uniform(300, D, seed=833, lo=-4.0, hi=4.0)])
    tr, tq = torch.from_numpy(refs).cuda(), torch.from_numpy(q).cuda()
    ctx.set_option(frnn.FRNN_OPT_GRID_AXES, axes)
    try:
        g = ctx.build_grid(tr, 0.125)
        got = ctx.query(g, tq, 0.125, 40, self_query=False, path="grid")
        ctx.sync()
        _same(got, oracle.frnn(q, refs, 0.125, 40))
        got = ctx.query(g, tq, 0.06, 40, self_query=False, path="grid")   # a smaller radius than the grid's
        ctx.sync()
        _same(got, oracle.frnn(q, refs, 0.06, 40))
    finally:
        ctx.set_option(frnn.FRNN_OPT_GRID_AXES, 0)


def test_batches_mix_half_cells_and_row_tasks(ctx):
    # D = 9: events of up to 16,384 points take row tasks, larger ones half cells
    import torch
    ev = [synth.event_mix(n, 9, (840, n)) for n in (300, 17001, 5000, 20000, 1, 0)]
    outs = ctx.query_batched([torch.from_numpy(p.reshape(-1, 9)).cuda() for p in ev], 0.1, 24, path="grid")
    ctx.sync()
    for p, o in zip(ev, outs):
        rows = np.arange(0, len(p), max(1, len(p) // 1500))
        if len(p):
            _same(tuple(x[torch.from_numpy(rows).cuda()] for x in o), oracle.self_query(p, 0.1, 24, rows=rows))


@pytest.mark.parametrize("size", [40, 100, 129, 140])
@pytest.mark.parametrize("budget", [0, 1 << 28])
def test_long_rows_beyond_the_pool(size, budget):
    # every row is longer than the lists; from 100 points a cluster on the
    # compact rows' pool (32 entries a query) runs out, from 130 the scratch
    import torch
    from paper_2609_31980_gb300 import frnn
    p = synth.clustered(30, size, 40, 8, 0.01, seed=850 + size)
    t = torch.from_numpy(p).cuda()
    for K in (129, 400):
        want = oracle.self_query(p, 0.1, K)
        with frnn.Context(budget_bytes=budget) as ctx:
            g = ctx.build_grid(t, 0.1)
            got = ctx.query(g, t, 0.1, K, path="grid")
            ctx.sync()
            _same(got, want)
            off, ci, cd, deg = ctx.query_csr(g, t, 0.1, K, degree=True)
            ctx.sync()
        keep = np.arange(K)[None, :] < want[0][:, None]
        np.testing.assert_array_equal(np.diff(off.cpu().numpy()), want[0])
        np.testing.assert_array_equal(ci.cpu().numpy(), want[1][keep])
        np.testing.assert_array_equal(cd.cpu().numpy().view(np.uint32), want[2][keep].view(np.uint32))
        np.testing.assert_array_equal(deg.cpu().numpy(), want[3])
