"""The tensor-core path on the automatic grids, whose half cells its tiles do not
walk: rows against the oracle (self, cross-set and compact queries, rebuilds,
batches, a caller's graph, a tight memory budget), and the time against the same
path on three requested axes."""
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


def _pts(n, D, seed):
    return synth.clustered(n // 50, 40, n - n // 50 * 40, D, 0.01, seed=seed)


@pytest.mark.parametrize("n,D,r,K", [(1, 8, 0.1, 8), (2001, 8, 0.1, 64), (4999, 8, 0.1, 64), (5000, 8, 0.1, 64), (16_385, 9, 0.1, 64),
                                     (20_000, 12, 0.12, 200), (33_001, 16, 0.12, 64), (40_000, 13, 0.12, 20)])
@pytest.mark.parametrize("axes", [0, 1])
def test_rows_on_the_automatic_grid(n, D, r, K, axes):
    import torch
    from paper_2609_31980_gb300 import frnn
    sets = [_pts(n, D, 80 + i) for i in range(2)]
    with frnn.Context() as ctx:
        ctx.set_option(frnn.FRNN_OPT_GRID_AXES, axes)
        g = None
        for p in (sets[0], sets[1], sets[0][:max(1, n // 2)].copy()):
            rows = np.arange(0, len(p), 1 + len(p) // 1500)
            want = oracle.self_query(p, r, K, rows=rows)
            t = torch.from_numpy(p).cuda()
            g = ctx.build_grid(t, r, grid=g)
            for path in ("tc", "grid", "tc"):
                _same(ctx.query(g, t, r, K, path=path), want, rows)
            off, ci, cd, deg = (x.cpu().numpy() for x in ctx.query_csr(g, t, r, K, path="tc", degree=True))
            np.testing.assert_array_equal(deg[rows], want[3])
            for k, row in enumerate(rows):
                c = want[0][k]
                assert off[row + 1] - off[row] == c
                np.testing.assert_array_equal(ci[off[row]:off[row + 1]], want[1][k, :c])
                np.testing.assert_array_equal(cd[off[row]:off[row + 1]].view(np.uint32), want[2][k, :c].view(np.uint32))
            q = sets[1][::3].copy()
            _same(ctx.query(g, torch.from_numpy(q).cuda(), r, K, self_query=False, path="tc"),
                  oracle.frnn(q[:300], p, r, K), slice(0, 300))
            ctx.sync()


def test_a_non_finite_point_is_reported_once():
    import torch
    from paper_2609_31980_gb300 import frnn
    p = _pts(20_000, 9, 84)
    p[777, 3] = np.nan
    t = torch.from_numpy(p).cuda()
    with frnn.Context() as ctx:
        g = ctx.build_grid(t, 0.1)
        with pytest.raises(frnn.FrnnError):
            ctx.sync()
        c, i, _ = ctx.query(g, t, 0.1, 16, path="tc")
        ctx.sync()
        assert int(c.abs().sum()) == 0 and bool((i == -1).all())


def test_batches_on_automatic_grids():
    import torch
    from paper_2609_31980_gb300 import frnn
    for D in (8, 12):
        ps = [_pts(n, D, 85 + n % 7) for n in (20_001, 17_000, 300, 40_000)]
        ts = [torch.from_numpy(p).cuda() for p in ps]
        with frnn.Context() as ctx:
            for graph in (0, 1):
                ctx.set_option(frnn.FRNN_OPT_USE_GRAPH, graph)
                outs = ctx.query_batched(ts, 0.1, 64, path="tc")
                ctx.sync()
                for p, o in zip(ps, outs):
                    rows = np.arange(0, len(p), 1 + len(p) // 700)
                    _same(o, oracle.self_query(p, 0.1, 64, rows=rows), rows)


@pytest.mark.parametrize("rebuild", [False, True])
def test_in_a_callers_graph(rebuild):
    import torch
    from paper_2609_31980_gb300 import frnn
    n, D, r, K = 20_000, 12, 0.12, 64
    a, b = _pts(n, D, 86), _pts(n, D, 87)
    s = torch.cuda.Stream()
    with frnn.Context(stream=s) as ctx:
        with torch.cuda.stream(s):
            t = torch.from_numpy(a).cuda()
            g = ctx.build_grid(t, r)
            out = (torch.empty(n, dtype=torch.int32, device="cuda"),
                   torch.empty(n, K, dtype=torch.int32, device="cuda"),
                   torch.empty(n, K, dtype=torch.float32, device="cuda"))
            ctx.query(g, t, r, K, path="tc", out=out)
        s.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=s):
            if rebuild:
                ctx.build_grid(t, r, grid=g)
            ctx.query(g, t, r, K, path="tc", out=out)
        rows = np.arange(0, n, 17)
        for p in ((b, a) if rebuild else (a,)):
            with torch.cuda.stream(s):
                t.copy_(torch.from_numpy(p))
            s.synchronize()
            graph.replay()
            torch.cuda.synchronize()
            ctx.sync()
            _same(out, oracle.self_query(p, r, K, rows=rows), rows)


def test_a_budget_without_room_for_the_tiles_grid():
    import torch
    from paper_2609_31980_gb300 import frnn
    n, D, r, K = 20_000, 8, 0.1, 64
    p = _pts(n, D, 88)
    t = torch.from_numpy(p).cuda()
    rows = np.arange(0, n, 17)
    want = oracle.self_query(p, r, K, rows=rows)
    least = None
    for mb in np.arange(2.0, 12.0, 0.25):
        with frnn.Context(budget_bytes=int(mb * 2**20)) as ctx:
            try:
                g = ctx.build_grid(t, r)
            except frnn.FrnnError:
                continue
            least = least or mb
            if mb > least + 1:
                break
            _same(ctx.query(g, t, r, K, path="tc"), want, rows)
            _same(ctx.query(g, t, r, K, path="grid"), want, rows)
            ctx.sync()
    assert least is not None


@pytest.mark.parametrize("n,D", [(200_000, 8), (100_000, 12)])
def test_time_is_that_of_the_tensor_core_path(n, D):
    """Walking the half cells took 8 to 50 times the time on three axes."""
    import torch
    from paper_2609_31980_gb300 import frnn
    t = torch.from_numpy(synth.event_mix(n, D, seed=3, per_cluster=20, sigma=0.02)).cuda()
    ms = {}
    for naxes in (3, 0):
        with frnn.Context() as ctx:
            ctx.set_option(frnn.FRNN_OPT_GRID_NAXES, naxes)
            g = ctx.build_grid(t, 0.12)
            out = ctx.query(g, t, 0.12, 64, path="tc")
            half = [t[:n // 2], t[n // 2:]]
            outs = ctx.query_batched(half, 0.12, 64, path="tc")

            def timed(fn):
                best = float("inf")
                for _ in range(5):
                    e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
                    e[0].record()
                    fn()
                    e[1].record()
                    e[1].synchronize()
                    best = min(best, e[0].elapsed_time(e[1]))
                return best

            def step():
                ctx.build_grid(t, 0.12, grid=g)
                ctx.query(g, t, 0.12, 64, path="tc", out=out)
            ms[naxes] = timed(step), timed(lambda: ctx.query_batched(half, 0.12, 64, path="tc", outs=outs))
    assert ms[0][0] < 2.5 * ms[3][0] and ms[0][1] < 2.5 * ms[3][1], ms
