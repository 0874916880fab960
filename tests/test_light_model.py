"""The light engine's rules, restated in numpy and run against the oracle on the CPU: each row lists
its lightest edges (here few, so that the lists are often incomplete), phases relax the dirty nodes
within a window, a row stops at the largest dist, and rows whose unlisted edges could still matter
are relaxed whole.  dist and pred must be Algorithm 1's for every order of relaxation the rules allow."""
import numpy as np
import pytest

import graphgen

INF = 2**31 - 1


def bits_for(n):
    b = 1
    while (1 << b) < n:
        b += 1
    return b


def build_index(W, cap, partial):
    """Per row: up to cap packed edges ascending, and the smallest weight not listed.  With `partial` a
    weight may be listed for some of its edges only (as the kernel's cut at cap does), else whole
    weights are dropped (as its cut at the buffer does)."""
    n, b = W.shape[0], bits_for(W.shape[0])
    rows, hmin = [], []
    for u in range(n):
        e = sorted((int(W[u, v]) << b) | v for v in range(n) if v != u and W[u, v] < INF)
        keep = e[:cap]
        if not partial and len(e) > cap:
            keep = [x for x in keep if (x >> b) < (e[cap] >> b)]
        rows.append(keep)
        hmin.append(e[len(keep)] >> b if len(keep) < len(e) else INF)
    return rows, hmin


def solve(W, source, rows, hmin, delta, rng):
    n, b = W.shape[0], bits_for(W.shape[0])
    umask, wf = (1 << b) - 1, (1 << (32 - b)) - 1
    none = (1 << 64) - 1
    key = [none] * n
    key[source] = 0
    dirty, hdone, heavy = {source}, set(), 0
    has_in = [any(W[u, v] < INF for u in range(n) if u != v) for v in range(n)]
    dist = lambda v: key[v] >> 32

    def offer(u, du, w, v):
        assert w <= wf
        k = ((du + w) << 32) | ((wf - w) << b) | u
        if k < key[v]:
            if (k >> 32) < dist(v):
                dirty.add(v)
            key[v] = k

    while True:
        D = max([dist(v) if dist(v) < INF else (1 << 32) - 1 for v in range(n) if dist(v) < INF or has_in[v]])
        if dirty:
            T = min(dist(v) for v in dirty) + delta
            now = [v for v in dirty if dist(v) <= T]
            rng.shuffle(now)
            dirty -= set(now)
            for u in now:
                du = dist(u)
                for e in rows[u]:
                    if du + (e >> b) > D:
                        break
                    offer(u, du, e >> b, e & umask)
            continue
        pend = [u for u in range(n) if u not in hdone and dist(u) < INF and hmin[u] < INF and dist(u) + hmin[u] <= D]
        if not pend:
            break
        bound = min(dist(u) + hmin[u] for u in pend)
        for u in [u for u in pend if dist(u) < bound]:
            hdone.add(u)
            heavy += 1
            du = dist(u)
            for v in range(n):
                if v != u and W[u, v] < INF and du + int(W[u, v]) <= D:
                    offer(u, du, int(W[u, v]), v)
    d = np.array([dist(v) if dist(v) < INF else INF for v in range(n)], dtype=np.int64)
    p = np.array([key[v] & umask if dist(v) < INF and v != source else -1 for v in range(n)], dtype=np.int64)
    return d, p, heavy


@pytest.mark.parametrize("cap", [1, 3, 64])
@pytest.mark.parametrize("directed", [False, True])
def test_rules_match_the_oracle(orc, cap, directed):
    rng = np.random.default_rng(cap * 2 + directed)
    heavy_total = 0
    for trial in range(60):
        n = int(rng.integers(1, 24))
        whi = int(rng.choice([1, 2, 5, 60, (2**31 - 2) // max(n - 1, 1)]))
        m = int(rng.integers(0, n * 5 + 1))
        e = graphgen.random_edges(n, m, 1, whi, seed=1000 * cap + trial, directed=directed)
        W = orc.build_matrix(n, e.src, e.dst, e.w, directed)
        rows, hmin = build_index(W, cap, partial=bool(trial & 1))
        s = int(rng.integers(0, n))
        ref = orc.dijkstra(W, s)
        for delta in (0, 1, 2**30):
            d, p, heavy = solve(W, s, rows, hmin, delta, rng)
            heavy_total += heavy
            assert np.array_equal(d, ref[0]), (trial, n, delta)
            assert np.array_equal(p, ref[1]), (trial, n, delta)
    assert heavy_total > 0 or cap == 64  # short lists do fall back to whole rows
