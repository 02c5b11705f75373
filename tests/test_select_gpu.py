"""Rows the scans hand to the selection kernel (select.cu), against the oracle
bit for bit: degrees around its register sorts' widths (32, 64, 128, 256 keys),
around the first pass' buffer (224 entries before it is cut or handed on), with
K on both sides of the largest K the first pass cuts at (192), ties included.
"""
import numpy as np
import pytest

from oracle import oracle

pytestmark = pytest.mark.gpu

# cluster sizes: degree = size - 1
SIZES = (33, 34, 64, 65, 66, 128, 129, 130, 224, 225, 226, 257, 258, 300, 700)


def _clusters(D, seed):
    """One tight cluster per size, far apart; every fourth point of a cluster
    repeats an earlier one (equal distances, ordered by index)."""
    g = np.random.default_rng(seed)
    parts = []
    for c, n in enumerate(SIZES):
        p = g.uniform(-0.01, 0.01, size=(n, D))
        p[3::4] = p[:len(p[3::4])]
        p[:, -1] += c * 0.5
        parts.append(p)
    pts = np.concatenate(parts)
    return pts[g.permutation(len(pts))].astype(np.float32)


@pytest.mark.parametrize("D", [1, 3, 8, 12, 16])
@pytest.mark.parametrize("K", [40, 192, 193, 1024])
def test_long_rows_match_oracle(D, K):
    import torch
    from paper_2609_31980_gb300 import frnn
    pts = _clusters(D, 700 + D)
    r = 0.25
    wc, wi, wd, wdeg = oracle.self_query(pts, r, K)
    t = torch.from_numpy(pts).cuda()
    with frnn.Context() as ctx:
        for _ in range(2):   # the second query finds the counters cleared
            c, i, d = ctx.self_query(t, r, K, path="grid")
            ctx.sync()
            assert np.array_equal(c.cpu().numpy(), wc)
            assert np.array_equal(i.cpu().numpy(), wi)
            assert np.array_equal(d.cpu().numpy().view(np.uint32), wd.view(np.uint32))
        g = ctx.build_grid(t, r)
        off, ci, cd, deg = ctx.query_csr(g, t, r, K, degree=True)
        ctx.sync()
    off, ci, cd = off.cpu().numpy(), ci.cpu().numpy(), cd.cpu().numpy()
    assert np.array_equal(deg.cpu().numpy(), wdeg)
    assert np.array_equal(np.diff(off), wc)
    keep = np.arange(K)[None, :] < wc[:, None]
    assert np.array_equal(ci, wi[keep])
    assert np.array_equal(cd.view(np.uint32), wd[keep].view(np.uint32))
