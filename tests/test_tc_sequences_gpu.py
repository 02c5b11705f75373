"""Queries of several kinds on one grid, without a rebuild in between: rows that
outgrow the selection kernel's first pass (more than 224 neighbours, K > 192)
on the tensor-core path leave nothing behind in the grid's list of such rows
that a later query of the same grid would take for its own."""
import numpy as np
import pytest

from oracle import oracle

pytestmark = pytest.mark.gpu

SIZES = (20, 34, 130, 226, 300, 700)   # clusters; degree = size - 1


def _points(D):
    g = np.random.default_rng(40 + D)
    parts = []
    for c, n in enumerate(SIZES):
        p = g.uniform(-0.01, 0.01, size=(n, D))
        p[:, -1] += c * 0.5
        parts.append(p)
    pts = np.concatenate(parts)
    return pts[g.permutation(len(pts))].astype(np.float32)


@pytest.mark.parametrize("D", [8, 12])
@pytest.mark.parametrize("naxes", [0, 3, 5])
@pytest.mark.parametrize("K", [193, 1024])
def test_paths_take_turns_on_one_grid(D, naxes, K):
    import torch
    from paper_2609_31980_gb300 import frnn
    pts = _points(D)
    r = 0.25
    want = oracle.self_query(pts, r, K)
    keep = np.arange(K)[None, :] < want[0][:, None]
    t = torch.from_numpy(pts).cuda()
    with frnn.Context() as ctx:
        ctx.set_option(frnn.FRNN_OPT_GRID_NAXES, naxes)
        g = ctx.build_grid(t, r)

        def dense(path):
            c, i, d = (x.cpu().numpy() for x in ctx.query(g, t, r, K, path=path))
            np.testing.assert_array_equal(c, want[0])
            np.testing.assert_array_equal(i, want[1])
            np.testing.assert_array_equal(d.view(np.uint32), want[2].view(np.uint32))

        def compact(path):
            off, i, d, deg = (x.cpu().numpy() for x in ctx.query_csr(g, t, r, K, path=path, degree=True))
            np.testing.assert_array_equal(deg, want[3])
            np.testing.assert_array_equal(np.diff(off), want[0])
            np.testing.assert_array_equal(i, want[1][keep])
            np.testing.assert_array_equal(d.view(np.uint32), want[2][keep].view(np.uint32))

        def count_only(path):   # the list stays for a fill pass that never runs
            off = torch.empty(len(pts) + 1, dtype=torch.int64, device="cuda")
            n = frnn._i64(0)
            st = frnn.frnn_query_csr_count(ctx.handle, g.handle, t.data_ptr(), len(pts), r, K,
                                           frnn.PATHS[path] | frnn.FRNN_SELF_QUERY, off.data_ptr(), None,
                                           frnn.ctypes.byref(n))
            assert st == 0 and n.value == int(want[0].sum())

        # (thirty rounds of a list that is never cleared would also overrun it)
        for _ in range(30):
            dense("tc")
        for step, path in ((dense, "grid"), (dense, "tc"), (compact, "grid"), (compact, "tc"), (dense, "grid"),
                           (count_only, "tc"), (dense, "grid"), (count_only, "grid"), (dense, "tc"),
                           (count_only, "tc"), (compact, "tc"), (dense, "tc"), (compact, "grid")):
            step(path)
        ctx.sync()
