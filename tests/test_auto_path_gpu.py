"""FRNN_PATH_AUTO on grids requested with up to three axes: either side of the
lines above which it takes the tensor-core path, against the grid scan."""
import pytest

from paper_2609_31980_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D,n,tc", [(10, 700_000, False), (11, 640_000, False), (12, 650_000, True),
                                    (13, 440_000, False), (13, 450_000, True)])
def test_auto_path_takes_the_faster_side(D, n, tc):
    import torch
    from paper_2609_31980_gb300 import frnn
    ctx = frnn.Context()
    try:
        ctx.set_option(frnn.FRNN_OPT_GRID_NAXES, 3)
        t = torch.from_numpy(synth.event_mix(n, D, seed=D, per_cluster=10, sigma=0.02)).cuda()
        assert t.shape[0] == n
        grid = ctx.build_grid(t, 0.1)
        ctx.set_option(frnn.FRNN_OPT_TC_SURVIVORS, 0)
        got = ctx.query(grid, t, 0.1, 12)
        assert (ctx.get_option(frnn.FRNN_OPT_TC_SURVIVORS) > 0) == tc
        for a, b in zip(got, ctx.query(grid, t, 0.1, 12, path="grid")):
            assert torch.equal(a, b)
    finally:
        ctx.close()
