"""The tensor-core path's epilogue (tc.cu) against the oracle bit for bit, where
it can go wrong: lists at the edges of the sort widths and of the list capacity,
more survivors in a group than a warp's buffer holds, ties of the truncated
sorting keys, tasks of few and of many chunks, both row writers, and compact
rows."""
import numpy as np
import pytest

from oracle import oracle

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


def _clusters(c, D, seed, n=3000):
    """Clusters of c points, all of them neighbours of one another, few enough
    apart in the gridded coordinates that a tile of queries meets several; every
    seventh point is a copy of another of its cluster."""
    g = np.random.default_rng(seed)
    m = max(1, n // c)
    centres = g.random((m, D), dtype=np.float32)
    p = np.repeat(centres, c, 0) + np.float32(0.002) * g.standard_normal((m * c, D)).astype(np.float32)
    dup = np.arange(0, m * c - 1, 7)
    same = dup // c == (dup + 1) // c
    p[dup[same] + 1] = p[dup[same]]
    return p.astype(np.float32)


@pytest.mark.parametrize("D", [8, 11, 12, 13, 16])
@pytest.mark.parametrize("c", [2, 9, 16, 17, 18, 30, 31, 32, 33, 90])
def test_list_lengths(ctx, D, c):
    import torch
    p = _clusters(c, D, 100 * D + c)
    t = torch.from_numpy(p).cuda()
    for K in (32, 35):   # 16-byte and 4-byte row writes
        _same(ctx.self_query(t, 0.05, K, path="tc"), oracle.self_query(p, 0.05, K))


@pytest.mark.parametrize("n", [1, 2, 31, 127, 129, 1024])
def test_one_row_of_cells(ctx, n):
    """All points in one cell of every axis but the fastest: tasks of one chunk
    up to tasks of eight, and almost every pair a survivor."""
    import torch
    g = np.random.default_rng(n)
    p = (g.random((n, 8), dtype=np.float32) * np.float32(0.1)).astype(np.float32)
    p[:, 7] = g.random(n, dtype=np.float32)
    _same(ctx.self_query(torch.from_numpy(p).cuda(), 0.2, 16, path="tc"), oracle.self_query(p, 0.2, 16))


def test_outputs_off_a_16_byte_boundary(ctx):
    import torch
    p = _clusters(20, 12, 5)
    n, K = len(p), 32
    t = torch.from_numpy(p).cuda()
    i = torch.empty(n * K + 1, dtype=torch.int32, device="cuda")[1:].view(n, K)
    d = torch.empty(n * K + 1, dtype=torch.float32, device="cuda")[1:].view(n, K)
    c = torch.empty(n, dtype=torch.int32, device="cuda")
    grid = ctx.build_grid(t, 0.05)
    _same(ctx.query(grid, t, 0.05, K, path="tc", out=(c, i, d)), oracle.self_query(p, 0.05, K))
