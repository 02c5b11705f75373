"""Two contexts in two host threads, as the header allows: the sizes one of them
works on change nothing for the other (a kernel's shared-memory limit belongs
to the function, not to the call that set it)."""
import threading

import numpy as np
import pytest

from oracle import oracle
from paper_2609_31980_gb300 import synth

pytestmark = pytest.mark.gpu


def _rows(D, seed):
    """A cluster whose rows outgrow the selection kernel's first pass."""
    g = np.random.default_rng(seed)
    return g.uniform(-0.01, 0.01, size=(400, D)).astype(np.float32)


@pytest.mark.parametrize("what", ["build", "select"])
def test_threads_with_sets_of_different_sizes(what):
    import torch
    from paper_2609_31980_gb300 import frnn
    if what == "build":   # one-launch builds of 135 KB and of 1 KB shared memory
        jobs = [(synth.clustered(400, 40, 32_768 - 16_000, 16, 0.01, seed=3), 0.1, 16, 300),
                (synth.clustered(2, 20, 10, 1, 0.01, seed=4), 0.1, 16, 900)]
    else:                 # second selection passes of 2,048 and of 512 keys a warp
        jobs = [(_rows(8, 5), 0.25, 1024, 300), (_rows(8, 6), 0.25, 193, 300)]
    go = threading.Barrier(len(jobs))
    errors = []

    def work(p, r, K, reps):
        try:
            s = torch.cuda.Stream()
            want = oracle.self_query(p, r, K, rows=np.arange(0, len(p), 1 + len(p) // 400))
            with torch.cuda.stream(s):
                t = torch.from_numpy(p).cuda()
                out = (torch.empty(len(p), dtype=torch.int32, device="cuda"),
                       torch.empty(len(p), K, dtype=torch.int32, device="cuda"),
                       torch.empty(len(p), K, dtype=torch.float32, device="cuda"))
            s.synchronize()
            with frnn.Context(stream=s) as ctx:
                grid = None
                go.wait(60)
                for _ in range(reps):
                    grid = ctx.build_grid(t, r, grid=grid)
                    ctx.query(grid, t, r, K, out=out)
                ctx.sync()
            got = [x.cpu().numpy()[::1 + len(p) // 400] for x in out]
            for a, b in zip(got, want):
                np.testing.assert_array_equal(a.view(np.uint32), b.view(np.uint32))
        except BaseException as e:   # noqa: BLE001 (reported by the main thread)
            errors.append(e)
            go.abort()

    threads = [threading.Thread(target=work, args=j) for j in jobs]
    for th in threads:
        th.start()
    for th in threads:
        th.join(300)
        assert not th.is_alive()
    assert not errors, errors
