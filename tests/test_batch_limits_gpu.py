"""Batches near the limits that they were always accepted within: 2^30 cells over
all events (16,385 entries for a small one), and a memory budget that just
holds the batch with one entry more than its cells an event."""
import numpy as np
import pytest

from oracle import oracle

pytestmark = pytest.mark.gpu


def _events(sizes, D, seed):
    g = np.random.default_rng(seed)
    return [g.uniform(0, 0.3, size=(n, D)).astype(np.float32) for n in sizes]


def _check(outs, evs, r, K, which):
    for e in which:
        want = oracle.self_query(evs[e], r, K)
        for a, b in zip(outs[e], want):
            np.testing.assert_array_equal(a.cpu().numpy().view(np.uint32), b.view(np.uint32))


@pytest.mark.parametrize("n_events", [52_427, 52_429, 65_531])
def test_many_small_events(n_events):
    import torch
    from paper_2609_31980_gb300 import frnn
    D, r, K = 3, 0.2, 4
    sizes = [1 + e % 7 for e in range(n_events)]
    evs = _events(sizes, D, 9)
    off = np.concatenate([[0], np.cumsum(sizes)])
    flat = torch.from_numpy(np.concatenate(evs)).cuda()
    c = torch.empty(off[-1], dtype=torch.int32, device="cuda")
    i = torch.empty(off[-1], K, dtype=torch.int32, device="cuda")
    d = torch.empty(off[-1], K, dtype=torch.float32, device="cuda")
    cut = lambda x: [x[off[e]:off[e + 1]] for e in range(n_events)]   # noqa: E731
    with frnn.Context() as ctx:
        outs = ctx.query_batched(cut(flat), r, K, outs=list(zip(cut(c), cut(i), cut(d))))
        ctx.sync()
        _check(outs, evs, r, K, list(range(0, n_events, 97)) + [n_events - 1])


def test_one_more_event_than_the_limit_is_refused():
    import torch
    from paper_2609_31980_gb300 import frnn
    t = torch.zeros(1, 3, device="cuda")
    out = (torch.empty(1, dtype=torch.int32, device="cuda"), torch.empty(1, 4, dtype=torch.int32, device="cuda"),
           torch.empty(1, 4, device="cuda"))
    n = 2**30 // 16_385 + 1
    with frnn.Context() as ctx:
        with pytest.raises(frnn.FrnnError) as e:
            ctx.query_batched([t] * n, 0.1, 4, outs=[out] * n)
        assert e.value.status == frnn.FRNN_ERR_INVALID_ARG


@pytest.mark.parametrize("D", [3, 8, 12])
@pytest.mark.parametrize("n_events", [1, 3, 200, 2000])
def test_batch_that_just_fits_its_budget(D, n_events):
    import torch
    from paper_2609_31980_gb300 import frnn
    r, K = 0.2, 8
    sizes = [1 + (37 * e) % 60 for e in range(n_events)]
    evs = _events(sizes, D, 10)
    # 232-byte headers, boxes, rows of whole 16 bytes, six words a slot, one
    # entry more than 16,384 cells, scan totals
    dp = (D + 3) // 4 * 4
    slots, cells = sum(n + 1 for n in sizes), 16_385 * n_events
    budget = (232 * n_events + 16 * (n_events + 1) + 4 * 34 * 32 * n_events + (slots + 512) * 4 * dp + slots * 24 +
              4 * cells + 4 * (cells // 2048 + 1) + 64 * 1024 + 16 * 256)
    ts = [torch.from_numpy(p).cuda() for p in evs]
    with frnn.Context(budget_bytes=budget) as ctx:
        outs = ctx.query_batched(ts, r, K)
        ctx.sync()
        _check(outs, evs, r, K, range(0, n_events, 1 + n_events // 60))
