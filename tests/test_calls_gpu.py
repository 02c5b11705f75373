"""What the library asks of the CUDA runtime, seen through a copy of it whose
runtime calls are listed (cuda_calls.cpp): run in child processes that load
that copy in place of the library."""
import os
import subprocess
import sys
import textwrap

import pytest

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
WRAPPED = ("cudaMalloc", "cudaMemsetAsync", "cudaMemcpyAsync", "cudaLaunchKernelExC")

PRELUDE = """
import ctypes, sys
import numpy as np
import torch
real = ctypes.CDLL
ctypes.CDLL = lambda p, *a, **k: real(sys.argv[1] if str(p).endswith("libfrnn.so") else p, *a, **k)
from oracle import oracle
from paper_2609_31980_gb300 import frnn, synth
lib = frnn._lib
lib.calls_bytes.restype = ctypes.c_size_t
def calls():
    return [(lib.calls_kind(i), lib.calls_bytes(i)) for i in range(lib.calls_count())]
def same(got, p, r, K):
    rows = np.arange(0, len(p), 1 + len(p) // 500)
    want = oracle.self_query(p, r, K, rows=rows)
    for a, b in zip((x.cpu().numpy()[rows] for x in got), want):
        assert np.array_equal(a.view(np.uint32), b.view(np.uint32))
"""


@pytest.fixture(scope="module")
def listed_lib(tmp_path_factory):
    from paper_2609_31980_gb300 import build
    d = tmp_path_factory.mktemp("calls")
    obj, so = str(d / "cuda_calls.o"), str(d / "listed.so")
    subprocess.run([build._nvcc(), "-O2", "-std=c++17", "-Xcompiler", "-fPIC", "-c",
                    os.path.join(HERE, "cuda_calls.cpp"), "-o", obj], check=True)
    objs = [os.path.join(build.BUILD_DIR, os.path.basename(s)[:-3] + ".o") for s in build.sources()]
    wraps = [f for w in WRAPPED for f in ("-Xlinker", f"--wrap={w}")]
    subprocess.run([build._nvcc(), *build.ARCH, "-shared", "-o", so, *objs, obj, *wraps, "-lpthread"], check=True)
    return so


def _child(so, code):
    r = subprocess.run([sys.executable, "-c", PRELUDE + textwrap.dedent(code), so], cwd=ROOT, timeout=300,
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-4000:]


def test_small_sets_build_without_large_clusters(listed_lib):
    """A device that cannot place a cluster of sixteen CTAs refuses the
    one-launch build: the separate kernels build the set, no error stays."""
    _child(listed_lib, """
        lib.calls_refuse_clusters(1)
        with frnn.Context() as ctx:
            for n, D, r, K in ((1, 3, 0.1, 8), (3000, 3, 0.08, 32), (20_000, 8, 0.1, 64), (9_001, 12, 0.12, 64)):
                p = synth.clustered(n // 50, 40, n - n // 50 * 40, D, 0.01, seed=70)
                t = torch.from_numpy(p).cuda()
                lib.calls_reset()
                g = ctx.build_grid(t, r)
                same(ctx.query(g, t, r, K), p, r, K)
                same(ctx.query(g, t, r, K, path="grid"), p, r, K)
                q = torch.from_numpy(p[:max(1, n // 3)].copy()).cuda()
                c, i, d = (x.cpu().numpy() for x in ctx.query(g, q, r, K, self_query=False))
                rows = np.arange(0, len(q), 1 + len(q) // 500)
                want = oracle.frnn(p[rows], p, r, K)
                assert np.array_equal(c[rows], want[0]) and np.array_equal(i[rows], want[1])
                assert np.array_equal(d[rows].view(np.uint32), want[2].view(np.uint32))
                ctx.sync()
                assert sum(k == 4 for k, _ in calls()) == 2, calls()
        """)


def test_compact_queries_clear_the_pool_only_when_they_use_it(listed_lib):
    """Rows past the staging width go to a pool in calls that keep more than
    128 neighbours: only those clear its counter."""
    _child(listed_lib, """
        p = synth.clustered(500, 40, 20_000, 8, 0.01, seed=71)
        t = torch.from_numpy(p).cuda()
        with frnn.Context() as ctx:
            g = ctx.build_grid(t, 0.1)
            for K in (1000, 64, 128, 129, 64):
                ctx.query_csr(g, t, 0.1, K)
                ctx.sync()
                lib.calls_reset()
                g = ctx.build_grid(t, 0.1, grid=g)
                ctx.query_csr(g, t, 0.1, K)
                ctx.self_query_host_csr(p, 0.1, K)
                ctx.self_query_host_csr(p, 0.1, K)
                clears = [n for k, n in calls() if k == 2 and n == 8]
                assert len(clears) == (3 if K > 128 else 0), (K, calls())
        """)


def test_compact_budget_holds_the_staging_rows_alone(listed_lib):
    """Under a memory budget there is no pool: the staging of a compact query
    is its counts, its rows of 32 and the scan totals, and no byte more."""
    _child(listed_lib, """
        n, D = 20_000, 8
        p = synth.clustered(500, 40, 0, D, 0.01, seed=72)
        t = torch.from_numpy(p).cuda()
        al = lambda x: (x + 255) // 256 * 256
        stage = al(4 * n) + 2 * al(128 * n) + al(8 * (-(-n // 8192)))
        for K in (64, 200):
            with frnn.Context(budget_bytes=64 << 20) as ctx:
                lib.calls_reset()
                g = ctx.build_grid(t, 0.1)
                ctx.query_csr(g, t, 0.1, K)
                ctx.sync()
                assert (1, stage) in calls(), (K, stage, calls())
        """)


def test_serving_allocates_before_the_first_request(listed_lib):
    """Every slot's workspace, the scan's scratch of calls that keep more than
    128 neighbours included, is made before the loop copies its first input."""
    _child(listed_lib, """
        ev = [synth.clustered(100, 40, 1000, 8, 0.01, seed=73 + i) for i in range(6)]
        with frnn.Context() as ctx:
            lib.calls_reset()
            outs, lat, st = ctx.serve(ev, [0.0] * len(ev), 0.1, 200, slots=2, max_batch=2)
            kinds = [k for k, n in calls()]
            copy = next(i for i, (k, n) in enumerate(calls()) if k == 3 and n == ev[0].nbytes)
            assert 1 in kinds[:copy] and 1 not in kinds[copy:], calls()
            for p, o in zip(ev, outs):
                same([torch.from_numpy(x) for x in o], p, 0.1, 200)
        """)


def test_compact_queries_without_long_rows_launch_no_second_selection(listed_lib):
    """Search, its selection, offsets, gather: nothing more when the count pass
    left no row to the selection, whatever K; the rows when it did."""
    _child(listed_lib, """
        for D, n in ((3, 3000), (8, 3000), (12, 3000), (8, 20_000)):
            p = synth.clustered(n // 50, 10, n - n // 50 * 10, D, 0.01, seed=75)
            long = p.copy()
            long[:700] = long[0] + np.random.default_rng(1).uniform(-1e-3, 1e-3, (700, D)).astype(np.float32)
            with frnn.Context() as ctx:
                for K in (64, 200):
                    for pts, r in ((p, 0.02), (long, 0.02), (p, 0.02)):
                        t = torch.from_numpy(pts).cuda()
                        g = ctx.build_grid(t, r)
                        ctx.query(g, t, r, K)      # (per-build preparation)
                        ctx.query_csr(g, t, r, K)
                        ctx.sync()
                        lib.calls_reset()
                        off, i, d, _ = ctx.query_csr(g, t, r, K)
                        launches = sum(k == 5 for k, _ in calls())
                        memsets = sum(k == 2 for k, _ in calls())
                        ctx.sync()
                        c = np.diff(off.cpu().numpy())
                        rows = np.arange(0, n, 7)
                        want = oracle.self_query(pts, r, K, rows=rows)
                        assert np.array_equal(c[rows], want[0])
                        off, i, d = off.cpu().numpy(), i.cpu().numpy(), d.cpu().numpy()
                        for k, row in enumerate(rows):
                            assert np.array_equal(i[off[row]:off[row + 1]], want[1][k, :want[0][k]])
                        half = g.scan()["scan"] in ("half cells", "wide cells")
                        assert memsets == (1 if half and K > 128 else 0), (D, n, K, calls())
                        parts = 2 if n > 8192 else 0
                        if pts is p:
                            assert launches == 4 + parts, (D, n, K, launches)
                        else:
                            assert launches > 4 + parts, (D, n, K, launches)
        """)
