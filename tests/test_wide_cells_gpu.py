"""Automatic grids whose axes hold only a few cells (radii of a tenth of the
extent and more): plain cells over four or five axes in place of half cells, and
the half-cell scan's way of searching them, against the oracle bit for bit and in
time against the scans of requested axes."""
import ctypes

import numpy as np
import pytest

from oracle import oracle
from paper_2609_31980_gb300 import synth

pytestmark = pytest.mark.gpu


def _same(got, want, rows=slice(None)):
    got = [x.cpu().numpy()[rows] for x in got]
    np.testing.assert_array_equal(got[0], want[0])
    np.testing.assert_array_equal(got[1], want[1])
    np.testing.assert_array_equal(got[2].view(np.uint32), want[2].view(np.uint32))


def _points(n, D, seed, lattice):
    g = np.random.default_rng(seed)
    p = g.uniform(0, 1, size=(n, D))
    p[:n // 20] = p[0] + g.uniform(-0.05, 0.05, size=(n // 20, D))   # rows past the lists
    if lattice:   # many equal distances, points on the cells' edges
        p = np.round(p * 8) / 8
    p[3::50] = p[:len(p[3::50])]
    return p.astype(np.float32)


# n: one chunk, ragged chunks, past the row-task default of D >= 9
@pytest.mark.parametrize("D", [5, 6, 7, 8, 9, 10, 11, 12, 13, 16])
@pytest.mark.parametrize("n,r,K", [(17_001, 0.3, 64), (17_003, 0.17, 12), (16_500, 0.3, 200)])
def test_rows_on_few_cells(D, n, r, K):
    import torch
    from paper_2609_31980_gb300 import frnn
    p, q = _points(n, D, 90 + D, K == 12), _points(n, D, 91 + D, K == 12)[::7].copy()
    rows = np.arange(0, n, 29)
    want = oracle.self_query(p, r, K, rows=rows)
    t, tq = torch.from_numpy(p).cuda(), torch.from_numpy(q).cuda()
    with frnn.Context() as ctx:
        for axes in (0, 1):
            ctx.set_option(frnn.FRNN_OPT_GRID_AXES, axes)
            g = ctx.build_grid(t, r)
            assert g.scan()["scan"] == "wide cells", g.scan()
            for _ in range(2):
                _same(ctx.query(g, t, r, K), want, rows)
        _same(ctx.query(g, t, 0.7 * r, K), oracle.self_query(p, np.float32(0.7 * r), K, rows=rows), rows)
        _same(ctx.query(g, tq, r, K, self_query=False), oracle.frnn(q[::5], p, r, K), slice(None, None, 5))
        if D >= 8:
            _same(ctx.query(g, t, r, K, path="tc"), want, rows)
        off, ci, cd, deg = (x.cpu().numpy() for x in ctx.query_csr(g, t, r, K, degree=True))
        ctx.sync()
        np.testing.assert_array_equal(deg[rows], want[3])
        for k, row in enumerate(rows):
            c = want[0][k]
            assert off[row + 1] - off[row] == c
            np.testing.assert_array_equal(ci[off[row]:off[row + 1]], want[1][k, :c])
            np.testing.assert_array_equal(cd[off[row]:off[row + 1]].view(np.uint32), want[2][k, :c].view(np.uint32))


@pytest.mark.parametrize("D", [5, 8])
@pytest.mark.parametrize("n", [1, 2, 15, 17, 700, 3001])
def test_small_sets(D, n):
    import torch
    from paper_2609_31980_gb300 import frnn
    p = _points(max(n, 60), D, 7 * D + n, False)[:n].copy()
    with frnn.Context() as ctx:
        for r in (0.12, 0.25, 0.5, 2.0):
            t = torch.from_numpy(p).cuda()
            want = oracle.self_query(p, r, 40)
            g = ctx.build_grid(t, r)
            _same(ctx.query(g, t, r, 40), want)
            out = (torch.empty(n, dtype=torch.int32, device="cuda"), torch.empty(n, 40, dtype=torch.int32, device="cuda"),
                   torch.empty(n, 40, device="cuda"))
            torch.cuda.synchronize()
            assert frnn.frnn_self_query_noalloc(t.data_ptr(), n, D, ctypes.c_float(r), 40, *(x.data_ptr() for x in out),
                                                torch.cuda.current_stream().cuda_stream) == 0
            _same(out, want)
        ctx.sync()


def test_batch_of_both_kinds():
    import torch
    from paper_2609_31980_gb300 import frnn
    D, r, K = 8, 0.2, 32
    ps = [_points(9_000, D, 1, False), synth.clustered(300, 40, 1000, D, 0.01, seed=2) * np.float32(20),
          _points(50, D, 3, False), _points(30_001, D, 4, True)]
    ts = [torch.from_numpy(p).cuda() for p in ps]
    with frnn.Context() as ctx:
        for graph in (0, 1):
            ctx.set_option(frnn.FRNN_OPT_USE_GRAPH, graph)
            for _ in range(2):
                outs = ctx.query_batched(ts, r, K)
            ctx.sync()
            for p, o in zip(ps, outs):
                rows = np.arange(0, len(p), 1 + len(p) // 600)
                _same(o, oracle.self_query(p, r, K, rows=rows), rows)


@pytest.mark.parametrize("D,n,r", [(8, 60_000, 0.25), (12, 60_000, 0.3), (16, 40_000, 0.25)])
def test_time_of_a_dense_set(D, n, r):
    """Half cells took 2.3 to 4 times the row tasks' time on these sets."""
    import torch
    from paper_2609_31980_gb300 import frnn
    t = torch.from_numpy(synth.uniform(n, D, seed=5)).cuda()
    ms = {}
    for naxes in (4, 0):
        with frnn.Context() as ctx:
            ctx.set_option(frnn.FRNN_OPT_GRID_NAXES, naxes)
            g = ctx.build_grid(t, r)
            out = ctx.query(g, t, r, 32)
            best = float("inf")
            for _ in range(5):
                e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
                e[0].record()
                ctx.build_grid(t, r, grid=g)
                ctx.query(g, t, r, 32, out=out)
                e[1].record()
                e[1].synchronize()
                best = min(best, e[0].elapsed_time(e[1]))
            ms[naxes] = best
    assert ms[0] < 1.4 * ms[4], ms
