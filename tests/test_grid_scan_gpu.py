"""frnn_grid_scan: the grid as it is stored and the scan that searches it."""
import numpy as np
import pytest

from paper_2609_31980_gb300 import synth

pytestmark = pytest.mark.gpu


def test_scan_and_stored_cells():
    import torch
    from paper_2609_31980_gb300 import frnn
    event = synth.config2().points
    cases = (   # points, r, requested axes, cell multiple, scan, axes (None: the build's choice)
        (event, 0.1, 0, 0, "half cells", [3, 4, 5, 6, 7, 2]),
        (synth.uniform(20_000, 5, seed=1), 0.08, 0, 0, "half cells", None),
        (synth.uniform(20_000, 5, seed=1), 0.25, 0, 0, "wide cells", None),
        (synth.uniform(20_000, 12, seed=1), 0.3, 0, 0, "wide cells", None),
        (synth.uniform(4096, 3, seed=2), 0.05, 0, 0, "query per lane", [0, 1, 2]),
        (synth.uniform(4096, 3, seed=2), 0.05, 0, 2, "query per lane", [0, 1, 2]),
        (synth.uniform(2000, 8, seed=3), 0.1, 3, 0, "rows", [5, 6, 7]),
        (synth.uniform(2000, 8, seed=3), 0.1, 5, 0, "chunks", [3, 4, 5, 6, 7]),
        (synth.uniform(2000, 8, seed=3), 0.05, 0, 2, "half cells", None),
        (synth.clustered(400, 25, 3000, 12, 0.025, seed=4), 0.12, 0, 0, "rows", [8, 9, 10, 11]))
    with frnn.Context() as ctx:
        for pts, r, naxes, mult, scan, axes in cases:
            ctx.set_option(frnn.FRNN_OPT_GRID_NAXES, naxes)
            ctx.set_option(frnn.FRNN_OPT_CELL_MULT, mult)
            g = ctx.build_grid(torch.from_numpy(pts).cuda(), r)
            s, p = g.scan(), g.params()
            assert s["scan"] == scan and s["cells"] == int(np.prod(s["dims"])), (s, p)
            assert len(s["axes"]) == s["naxes"] == len(set(s["axes"]))
            assert axes is None or s["axes"] == axes, s
            if scan == "half cells":   # two by two along every axis but the first
                assert s["axes"][:p["naxes"]] == p["axes"]
                assert s["dims"][0] == p["dims"][0]
                assert s["dims"][1:p["naxes"]] == [(d + 1) // 2 for d in p["dims"][1:]]
            else:
                assert (s["axes"], s["dims"], s["cells"]) == (p["axes"], p["dims"], p["cells"])
            g.close()
