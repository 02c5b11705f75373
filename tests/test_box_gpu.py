"""The bounding boxes of the large build (k_bbox, build.cu), which reads each
event as one run of floats: every element of the run has to reach the minimum
and the maximum of its own coordinate, whatever the dimension, the alignment of
the input, the row and the number of floats past the last 16-byte piece."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_2609_31980_gb300 import frnn
    c = frnn.Context()
    yield c
    c.close()


def _at(p, offset):
    """p on the device, `offset` floats past a 16-byte boundary."""
    import torch
    buf = torch.empty(p.size + offset, dtype=torch.float32, device="cuda")
    t = buf[offset:].view(p.shape)
    t.copy_(torch.from_numpy(p))
    return t


@pytest.mark.parametrize("D", [1, 2, 3, 5, 6, 7, 8, 9, 12, 13, 16])
@pytest.mark.parametrize("offset", [0, 1, 2, 3])
def test_every_element_reaches_its_coordinate(ctx, D, offset):
    from paper_2609_31980_gb300 import frnn
    g = np.random.default_rng(10 * D + offset)
    n = 40_003
    p = g.random((n, D), dtype=np.float32)
    t = _at(p, offset)
    ctx.set_option(frnn.FRNN_OPT_GRID_AXES, 1)     # the widest coordinate
    ctx.set_option(frnn.FRNN_OPT_GRID_NAXES, 1)
    ctx.set_option(frnn.FRNN_OPT_CELL_MULT, 1)
    try:
        for j, row in enumerate([0, 1, 255, 256, 511, n - 2, n - 1, int(g.integers(n))]):
            k = int(g.integers(D))
            keep = float(t[row, k])
            t[row, k] = 3.0 if j % 2 else -2.0     # this coordinate is now 3 wide, the others 1
            grid = ctx.build_grid(t, 0.1)
            q = grid.params()
            assert q["axes"] == [k] and 28 <= q["dims"][0] <= 31, (row, k, q)
            grid.close()
            t[row, k] = float("nan") if j % 2 else float("inf")
            with pytest.raises(frnn.FrnnError):
                grid = ctx.build_grid(t, 0.1)
                ctx.sync()
            t[row, k] = keep
    finally:
        ctx.set_option(frnn.FRNN_OPT_GRID_AXES, 0)
        ctx.set_option(frnn.FRNN_OPT_GRID_NAXES, 0)
        ctx.set_option(frnn.FRNN_OPT_CELL_MULT, 0)


def test_events_of_one_block_share_a_run_only_with_themselves(ctx):
    """A CTA's build blocks cross event borders: each event's grid has to hold
    all of its points (a batch whose events lie far apart, against single
    queries)."""
    import torch
    g = np.random.default_rng(77)
    sizes = [1, 300, 255, 256, 257, 70_000, 3, 40_000, 513, 90_001]
    evs = [torch.from_numpy((g.random((s, 6), dtype=np.float32) + np.float32(3 * i))).cuda()
           for i, s in enumerate(sizes)]
    got = ctx.query_batched(evs, 0.12, 16)
    for t, (c, i, d) in zip(evs, got):
        for a, b in zip((c, i, d), ctx.self_query(t, 0.12, 16)):
            assert torch.equal(a, b)
