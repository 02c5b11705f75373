"""Builds and queries recorded into a caller's own CUDA graph: a call that would
have allocated its scratch takes the way without it, and a replay on new points
returns their rows."""
import numpy as np
import pytest

from oracle import oracle
from paper_2609_31980_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,D,r,K", [(3000, 3, 0.08, 32), (3000, 8, 0.1, 64), (3000, 8, 0.1, 200),
                                     (40_000, 8, 0.1, 200), (3000, 12, 0.12, 64)])
def test_build_and_query_in_a_callers_graph(n, D, r, K):
    import torch
    from paper_2609_31980_gb300 import frnn
    a, b = (synth.clustered(n // 50, 40, n - n // 50 * 40, D, 0.01, seed=s) for s in (1, 2))
    s = torch.cuda.Stream()
    ctx = frnn.Context(stream=s)
    try:
        with torch.cuda.stream(s):
            t = torch.from_numpy(a).cuda()
            grid = ctx.build_grid(t, r)
            ctx.query(grid, t, r, 16)                 # (a first call, of the kind that needs no scratch)
            out = (torch.empty(n, dtype=torch.int32, device="cuda"),
                   torch.empty(n, K, dtype=torch.int32, device="cuda"),
                   torch.empty(n, K, dtype=torch.float32, device="cuda"))
        s.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=s):
            ctx.build_grid(t, r, grid=grid)
            ctx.query(grid, t, r, K, out=out)
        rows = np.arange(0, n, 1 if n < 4000 else 37)
        for p in (b, a):
            with torch.cuda.stream(s):
                t.copy_(torch.from_numpy(p))
            s.synchronize()
            graph.replay()
            torch.cuda.synchronize()
            ctx.sync()
            want = oracle.self_query(p, r, K, rows=rows)
            got = [x.cpu().numpy()[rows] for x in out]
            np.testing.assert_array_equal(got[0], want[0])
            np.testing.assert_array_equal(got[1], want[1])
            np.testing.assert_array_equal(got[2].view(np.uint32), want[2].view(np.uint32))
    finally:
        ctx.close()
