"""Up to four dimensions, sets on both sides of the sizes where a query is given
one, four and eight lanes, with every cell multiple (3 to 125 neighbour rows
shared by the lanes): rows against the oracle, time against the row tasks."""
import numpy as np
import pytest

from oracle import oracle
from paper_2609_31980_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D", [1, 2, 3, 4])
@pytest.mark.parametrize("mult", [1, 2, 3])
@pytest.mark.parametrize("n", [31, 14_560, 14_600, 29_150, 29_190])
def test_rows(D, mult, n):
    import torch
    from paper_2609_31980_gb300 import frnn
    p = synth.uniform(n, D, seed=30 + D)
    p[5::40] = p[:len(p[5::40])]
    r = float((2.0 / n) ** (1 / D))
    rows = np.arange(0, n, 1 + n // 900)
    want = oracle.self_query(p, r, 24, rows=rows)
    t = torch.from_numpy(p).cuda()
    with frnn.Context() as ctx:
        ctx.set_option(frnn.FRNN_OPT_CELL_MULT, mult)
        g = ctx.build_grid(t, r)
        out = ctx.query(g, t, r, 24)
        ctx.sync()
    for a, b in zip((x.cpu().numpy()[rows] for x in out), want):
        np.testing.assert_array_equal(a.view(np.uint32), b.view(np.uint32))


@pytest.mark.parametrize("n", [12_000, 30_000, 50_000])
def test_time_of_fine_cells(n):
    """Cells of r / 2 at D = 4: every lane used to walk all 125 neighbour rows."""
    import torch
    from paper_2609_31980_gb300 import frnn
    t = torch.from_numpy(synth.uniform(n, 4, seed=5)).cuda()
    r = float((1.5 / n) ** 0.25)
    us = {}
    with frnn.Context() as ctx:
        for mult in (1, 2):
            ctx.set_option(frnn.FRNN_OPT_CELL_MULT, mult)
            g = ctx.build_grid(t, r)
            out = ctx.query(g, t, r, 32)
            best = float("inf")
            for _ in range(7):
                e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
                e[0].record()
                for _ in range(20):
                    ctx.build_grid(t, r, grid=g)
                    ctx.query(g, t, r, 32, out=out)
                e[1].record()
                e[1].synchronize()
                best = min(best, e[0].elapsed_time(e[1]) * 50)
            us[mult] = best
    assert us[2] < 1.9 * us[1], us
