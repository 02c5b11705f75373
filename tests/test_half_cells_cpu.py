"""Grids of half cells (EventHdr::half, query_half.cu), index logic on the CPU.

Along every gridded axis but the fastest two neighbouring cells share a stored
cell (coordinate >> 1), the low bit saying which half.  Checked here: the stored
cells a query visits hold every cell within +-1 of its own, each once, and none
outside the grid (lane l of the scan moves along axis a when bit a - 1 of l is
set; moves that would leave the grid are masked); the header's 2^36 / d
multiplier divides exactly; the row sort's truncated 32-bit keys with the
counting repair give the (d2, index) order."""
import itertools

import numpy as np
import pytest


@pytest.mark.parametrize("dims", [(5,), (6,), (1,), (2,), (3, 4), (1, 5), (4, 1, 3), (2, 3, 2, 5)])
def test_visited_cells_hold_the_neighbourhood(dims):
    sdims = [(d + 1) >> 1 for d in dims]
    for c in itertools.product(*[range(d) for d in dims]):
        bits = sum((x & 1) << a for a, x in enumerate(c))
        st = [x >> 1 for x in c]
        bad = 0
        for a, sd in enumerate(sdims):
            if (st[a] == sd - 1) if (bits >> a) & 1 else (st[a] == 0):
                bad |= 1 << a
        seen = []
        for lane in range(1 << len(dims)):
            if lane & bad:
                continue
            v = [st[a] + (((1 if (bits >> a) & 1 else -1)) if (lane >> a) & 1 else 0)
                 for a in range(len(dims))]
            assert all(0 <= v[a] < sdims[a] for a in range(len(dims)))
            seen.append(tuple(v))
        assert len(set(seen)) == len(seen)
        near = itertools.product(*[range(max(x - 1, 0), min(x + 1, d - 1) + 1) for x, d in zip(c, dims)])
        assert {tuple(y >> 1 for y in n) for n in near} <= set(seen)


def test_division_by_multiplier_is_exact():
    for d in range(1, 1025):
        mag = -(-(1 << 36) // d)
        top = (1 << 26) - 1
        v = {0, 1, d - 1, d, top, top - 1} | {k * d + o for k in (1, 7, top // d) for o in (-1, 0, 1)}
        for x in v:
            if 0 <= x <= top:
                assert (x * mag) >> 36 == x // d


def _network(P):
    p = 1
    while p < P:
        q = p
        while q >= 1:
            j = q % p
            for i in range(P):
                if i >= j and (i - j) % (2 * q) < q and i + q < P and i // (2 * p) == (i + q) // (2 * p):
                    yield i, i + q
            q //= 2
        p *= 2


def _sort_row(d2, idx, P):
    """sort_rows<P> on one row: the order of its entries."""
    n = len(d2)
    bits = d2.view(np.uint32)
    key = [[0] * P, [0] * P]
    for h in range(2):
        for i in range(P):
            e = h * P + i
            key[h][i] = (int(bits[e]) & ~31) | e if e < n else 0x80000000 | (e * 33)
        for a, b in _network(P):
            if key[h][a] > key[h][b]:
                key[h][a], key[h][b] = key[h][b], key[h][a]
    lo = [min(key[0][i], key[1][P - 1 - i]) for i in range(P)]
    hi = [max(key[1][i], key[0][P - 1 - i]) for i in range(P)]
    for k in (lo, hi):
        j = P // 2
        while j:
            for i in range(P):
                if not i & j and k[i] > k[i | j]:
                    k[i], k[i | j] = k[i | j], k[i]
            j //= 2
    k = lo + hi
    tied = any((a ^ b) < 32 for a, b in zip(k, k[1:]))
    order = [x & 31 for x in k[:n]]
    if tied:
        full = [(float(d2[e]), int(idx[e])) for e in order]
        out = [0] * n
        for e, f in zip(order, full):
            out[sum(g < f for g in full)] = e
        order = out
    return order


@pytest.mark.parametrize("P", [4, 8, 16])
def test_row_sort_gives_the_key_order(P):
    g = np.random.default_rng(40 + P)
    for n in range(0, 2 * P + 1):
        for kind in range(3):
            d2 = g.random(n, dtype=np.float32)
            if kind == 1:      # equal distances
                d2 = g.integers(0, 3, n).astype(np.float32)
            elif kind == 2:    # distances a few units in the last place apart
                d2 = (np.float32(0.5).view(np.uint32) + g.integers(0, 70, n).astype(np.uint32)).view(np.float32)
            idx = g.permutation(1000)[:n].astype(np.int32)
            order = _sort_row(d2, idx, P)
            assert order == sorted(range(n), key=lambda e: (float(d2[e]), int(idx[e])))
