"""The first tensor-core query of a set on a stream of its own, while the default
stream is busy: the new operands' zeroing, which goes there, is complete before
they are written."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from oracle import oracle
from paper_2609_31980_gb300 import synth

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def delay(tmp_path_factory):
    """30 ms of work on the default stream."""
    from paper_2609_31980_gb300 import build
    so = str(tmp_path_factory.mktemp("delay") / "early_producer.so")
    subprocess.run([build._nvcc(), *build.ARCH, "-O2", "-shared", "-Xcompiler", "-fPIC", "-o", so,
                    os.path.join(HERE, "early_producer.cu")], check=True)
    fn = ctypes.CDLL(so).produce
    fn.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_int64, ctypes.c_uint64, ctypes.c_void_p]

    def run():
        assert fn(None, None, 0, 30_000_000, None) == 0
    return run


@pytest.mark.parametrize("naxes", [0, 3])
@pytest.mark.parametrize("batch", [False, True])
def test_first_query_beside_a_busy_default_stream(delay, naxes, batch):
    import torch
    from paper_2609_31980_gb300 import frnn
    p = synth.clustered(400, 40, 4000, 12, 0.01, seed=9)
    rows = np.arange(0, len(p), 19)
    want = oracle.self_query(p, 0.12, 32, rows=rows)
    s = torch.cuda.Stream()   # (does not synchronise with the default stream)
    with torch.cuda.stream(s):
        t = torch.from_numpy(p).cuda()
        out = (torch.empty(len(p), dtype=torch.int32, device="cuda"),
               torch.empty(len(p), 32, dtype=torch.int32, device="cuda"),
               torch.empty(len(p), 32, dtype=torch.float32, device="cuda"))
    torch.cuda.synchronize()
    with frnn.Context(stream=s) as ctx:
        ctx.set_option(frnn.FRNN_OPT_GRID_NAXES, naxes)
        g = ctx.build_grid(t, 0.12)
        ctx.sync()
        delay()
        if batch:
            ctx.query_batched([t], 0.12, 32, path="tc", outs=[out])
        else:
            ctx.query(g, t, 0.12, 32, path="tc", out=out)
        ctx.sync()
        torch.cuda.synchronize()
    for a, b in zip((x.cpu().numpy()[rows] for x in out), want):
        np.testing.assert_array_equal(a.view(np.uint32), b.view(np.uint32))


def test_counters_are_reset_in_order_with_the_queries(delay):
    import torch
    from paper_2609_31980_gb300 import frnn
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        t = torch.from_numpy(synth.clustered(400, 40, 4000, 12, 0.01, seed=9)).cuda()
    torch.cuda.synchronize()
    with frnn.Context(stream=s) as ctx:
        ctx.set_option(frnn.FRNN_OPT_GRID_NAXES, 3)
        g = ctx.build_grid(t, 0.12)
        with torch.cuda.stream(s):
            out = ctx.query(g, t, 0.12, 64, path="tc")
        ctx.sync()
        delay()
        ctx.set_option(frnn.FRNN_OPT_TC_SURVIVORS, 0)
        ctx.query(g, t, 0.12, 64, path="tc", out=out)
        ctx.sync()
        torch.cuda.synchronize()
        # (clusters of 40: no row is cut to K, so the rows hold every accepted pair)
        assert ctx.get_option(frnn.FRNN_OPT_TC_ACCEPTED) == int(out[0].sum())
