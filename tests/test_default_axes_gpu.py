"""The default gridded axes from D = 9 on, by size and requested cell multiple."""
import numpy as np
import pytest

from oracle import oracle
from paper_2609_31980_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D", [9, 12])
@pytest.mark.parametrize("mult", [0, 1, 2, 3])
@pytest.mark.parametrize("n", [16_384, 16_385])
def test_cell_multiples_change_nothing_about_them(D, mult, n):
    import torch
    from paper_2609_31980_gb300 import frnn
    p = synth.clustered(n // 50, 40, n - n // 50 * 40, D, 0.01, seed=80)
    t = torch.from_numpy(p).cuda()
    rows = np.arange(0, n, 23)
    want = oracle.self_query(p, 0.12, 32, rows=rows)
    with frnn.Context() as ctx:
        ctx.set_option(frnn.FRNN_OPT_CELL_MULT, mult)
        g = ctx.build_grid(t, 0.12)
        assert g.scan()["scan"] == ("rows" if n <= 16_384 else "half cells"), g.scan()
        outs = [ctx.query(g, t, 0.12, 32), ctx.query_batched([t, t[:700]], 0.12, 32)[0]]
        ctx.sync()
        for o in outs:
            for a, b in zip((x.cpu().numpy()[rows] for x in o), want):
                np.testing.assert_array_equal(a.view(np.uint32), b.view(np.uint32))
