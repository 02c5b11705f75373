"""The one-launch build of small sets (build.cu, k_build_small) against the
oracle: its size limits and the CTAs' uneven shares, points that do not start on
a 16-byte boundary, rebuilds between the two builds in one grid, cross sets and
non-finite input."""
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


def _t(a, off=0):
    """The array on the GPU, its first element `off` floats into its storage."""
    import torch
    flat = torch.zeros(a.size + off, dtype=torch.float32, device="cuda")
    flat[off:] = torch.from_numpy(np.ascontiguousarray(a)).cuda().reshape(-1)
    return flat[off:].view(a.shape)


def _check(ctx, grid, t, p, r, K):
    import torch
    got = ctx.query(grid, t, r, K, path="grid")
    ctx.sync()
    rows = np.arange(0, len(p), max(1, len(p) // 700))
    at = torch.from_numpy(rows).cuda()
    want = oracle.self_query(p, r, K, rows=rows)
    c, i, d = (x[at].cpu().numpy() for x in got)
    np.testing.assert_array_equal(c, want[0])
    np.testing.assert_array_equal(i, want[1])
    np.testing.assert_array_equal(d.view(np.uint32), want[2].view(np.uint32))


@pytest.mark.parametrize("D", [1, 3, 8, 11, 16])
def test_sizes_in_one_grid(ctx, D):
    r = 0.02 if D <= 3 else 0.12
    grid = None
    for n in (32769, 32768, 32767, 16385, 16384, 1023, 17, 16, 15, 1, 33000):
        p = synth.uniform(n, D, seed=960 + n) if D <= 3 else synth.event_mix(n, D, 960 + n, per_cluster=15)
        t = _t(p, n % 4)
        grid = ctx.build_grid(t, r, grid=grid)
        _check(ctx, grid, t, p, r, 24)


def test_cross_sets_and_nonfinite_points(ctx):
    from paper_2609_31980_gb300 import frnn
    refs = synth.event_mix(12000, 8, 970)
    q = np.concatenate([refs[:500] + np.float32(0.01), synth.uniform(101, 8, 971, lo=-3, hi=3)])
    g = ctx.build_grid(_t(refs), 0.1)
    got = ctx.query(g, _t(q, 1), 0.1, 40, self_query=False, path="grid")
    ctx.sync()
    want = oracle.frnn(q, refs, 0.1, 40)
    for a, b in zip(got, want):
        np.testing.assert_array_equal(a.cpu().numpy(), b)
    for bad in (np.nan, np.inf, -np.inf):
        x = refs.copy()
        x[7777, 3] = bad
        t = _t(x)
        g = ctx.build_grid(t, 0.1)
        c, i, d = ctx.query(g, t, 0.1, 8, path="grid")
        with pytest.raises(frnn.FrnnError) as e:
            ctx.sync()
        assert e.value.status == -5
        assert int(c.sum()) == 0 and bool((i == -1).all())
        y = q.copy()
        y[3, 0] = bad
        ctx.query(ctx.build_grid(_t(refs), 0.1), _t(y), 0.1, 8, self_query=False, path="grid")
        with pytest.raises(frnn.FrnnError):
            ctx.sync()
    g = ctx.build_grid(_t(refs), 0.1)   # the context is usable afterwards
    _check(ctx, g, g.points, refs, 0.1, 40)
