"""Points written just before the call by a kernel that has already let its
successors start (programmatic dependent launch): every build reads them after
that kernel, whatever the buffer held before."""
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
def produce(tmp_path_factory):
    from paper_2609_31980_gb300 import build
    so = str(tmp_path_factory.mktemp("producer") / "early_producer.so")
    subprocess.run([build._nvcc(), *build.ARCH, "-O2", "-shared", "-Xcompiler", "-fPIC", "-o", so,
                    os.path.join(HERE, "early_producer.cu")], check=True)
    fn = ctypes.CDLL(so).produce
    fn.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_int64, ctypes.c_uint64, ctypes.c_void_p]

    def run(dst, src, stream):
        assert fn(dst.data_ptr(), src.data_ptr(), src.numel(), 3_000_000, stream.cuda_stream) == 0
    return run


def _check(got, p, r, K, q=None):
    rows = np.arange(0, len(p if q is None else q), 1 if len(p) < 4000 else 61)
    want = oracle.self_query(p, r, K, rows=rows) if q is None else oracle.frnn(q[rows], p, r, K)
    got = [x.cpu().numpy()[rows] for x in got]
    np.testing.assert_array_equal(got[0], want[0])
    np.testing.assert_array_equal(got[1], want[1])
    np.testing.assert_array_equal(got[2].view(np.uint32), want[2].view(np.uint32))


# one-launch builds, and the separate kernels
@pytest.mark.parametrize("n,D,r,K", [(3000, 3, 0.08, 32), (20_000, 8, 0.1, 64), (60_000, 3, 0.02, 32),
                                     (60_000, 8, 0.1, 64), (40_000, 12, 0.12, 64)])
@pytest.mark.parametrize("cross", [False, True])
def test_points_of_an_early_producer(produce, n, D, r, K, cross):
    import torch
    from paper_2609_31980_gb300 import frnn
    s = torch.cuda.Stream()
    sets = [synth.clustered(n // 50, 40, n - n // 50 * 40, D, 0.01, seed=60 + i) for i in range(3)]
    with torch.cuda.stream(s):
        srcs = [torch.from_numpy(p).cuda() for p in sets]
        ref = torch.from_numpy(sets[0]).cuda()
        buf = torch.zeros_like(ref)
    s.synchronize()
    with frnn.Context(stream=s) as ctx:
        out = tuple(torch.empty(sh, dtype=dt, device="cuda") for sh, dt in
                    (((n,), torch.int32), ((n, K), torch.int32), ((n, K), torch.float32)))
        grid = ctx.build_grid(ref, r)
        ctx.query(grid, ref, r, K, out=out)
        if cross:
            ctx.query(grid, buf, r, K, self_query=False, out=out)   # (its workspace)
        for p, src in zip(sets, srcs):
            s.synchronize()
            produce(buf, src, s)
            if cross:
                ctx.query(grid, buf, r, K, self_query=False, out=out)
            else:
                grid = ctx.build_grid(buf, r, grid=grid)
                ctx.query(grid, buf, r, K, out=out)
            ctx.sync()
            _check(out, sets[0] if cross else p, r, K, p if cross else None)
