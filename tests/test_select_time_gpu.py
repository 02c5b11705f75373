"""Rows that the selection kernel's first pass hands on (K > 192, more than 224
neighbours), all of them next to each other in its list: the second pass spreads
them over the chip."""
import numpy as np
import pytest

from oracle import oracle
from paper_2609_31980_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [31, 3000, 20_000])
def test_many_rows_of_the_second_pass(n):
    import torch
    from paper_2609_31980_gb300 import frnn
    p = synth.uniform(n, 3, seed=5)
    r = float(min(1.0, (1500 / n / 4.19) ** (1 / 3)))
    t = torch.from_numpy(p).cuda()
    ms = {}
    with frnn.Context() as ctx:
        g = ctx.build_grid(t, r)
        for K in (192, 300):
            best = float("inf")
            for _ in range(5):
                e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
                e[0].record()
                out = ctx.query(g, t, r, K)
                e[1].record()
                e[1].synchronize()
                best = min(best, e[0].elapsed_time(e[1]))
            ms[K] = best
            rows = np.arange(0, n, 1 + n // 300)
            want = oracle.self_query(p, r, K, rows=rows)
            for a, b in zip((x.cpu().numpy()[rows] for x in out), want):
                np.testing.assert_array_equal(a.view(np.uint32), b.view(np.uint32))
        ctx.sync()
    # (32 consecutive rows a warp, 3000 points: nine times)
    assert ms[300] < 4 * ms[192] + 0.05, ms
