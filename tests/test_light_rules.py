"""The light engine's rules as the library compiles them (dj_light_rules.h), run on the CPU: the stage that
relaxes rows whole ends on every matrix, whatever its rows leave unlisted, and keeps the answer."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

from test_light_model import INF, build_index

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2504_03667_gb300", "csrc")
NONE = 2**32 - 1

PROG = r"""
#include <cstddef>
#include "dj_light_rules.h"
extern "C" {
unsigned pending(unsigned dist, unsigned hmin, unsigned D) { return dj::light_pending(dist, hmin, D); }
unsigned below(unsigned hb, unsigned hmin_min) { return dj::light_below(hb, hmin_min); }
int in_place(size_t a, size_t b, size_t c) { return dj::edges_in_place((void*)a, (void*)b, (void*)c); }
int upload_in_place(size_t a) { return dj::in_place((void*)a); }
unsigned trial_word(unsigned u, unsigned listed, int has_edges, unsigned n) {
  return dj::light_trial_word(u, listed, has_edges, n);
}
unsigned trial_source(unsigned word, unsigned n) { return dj::light_trial_source(word, n); }
int verdict(unsigned rows, unsigned guess, unsigned risky) { return dj::light_trial_verdict(rows, guess, risky); }
int risky(unsigned dist, unsigned hmin, unsigned D) { return dj::light_risky(dist, hmin, D); }
int few(int n, unsigned guess, int wmin) { return dj::light_few(n, guess, wmin); }
int needs_trial(unsigned hmin_min, unsigned wmin) { return dj::light_needs_trial(hmin_min, wmin); }
}
"""


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    d = tmp_path_factory.mktemp("rules")
    src, lib = d / "rules.cpp", d / "librules.so"
    src.write_text(PROG)
    subprocess.run([cxx, "-std=c++17", "-O1", "-fPIC", "-shared", "-I", CSRC, str(src), "-o", str(lib)], check=True)
    lib = ctypes.CDLL(str(lib))
    for f, args in ((lib.pending, 3), (lib.below, 2), (lib.needs_trial, 2), (lib.trial_word, 4), (lib.trial_source, 2),
                    (lib.verdict, 3), (lib.risky, 3), (lib.few, 3)):
        f.argtypes = [ctypes.c_uint32] * args
    lib.upload_in_place.argtypes = [ctypes.c_size_t]
    lib.in_place.argtypes = [ctypes.c_size_t] * 3
    for f in (lib.pending, lib.below, lib.trial_word, lib.trial_source):
        f.restype = ctypes.c_uint32
    return lib


def solve(W, s, rows, hmin, rules):
    """dist by the listed edges and whole rows; at most one round of whole rows per node."""
    n, b = W.shape[0], 1
    while (1 << b) < n:
        b += 1
    dist = [NONE] * n
    dist[s] = 0
    whole = set()
    has_in = [any(W[u, v] < INF for u in range(n) if u != v) for v in range(n)]
    for rounds in range(n + 2):
        dirty = list(range(n))
        while dirty:  # settle on the listed edges
            u = dirty.pop()
            if dist[u] == NONE:
                continue
            for e in rows[u]:
                v, c = e & ((1 << b) - 1), dist[u] + (e >> b)
                if c < dist[v]:
                    dist[v] = c
                    dirty.append(v)
        D = max(dist[v] if dist[v] != NONE else (NONE if has_in[v] else 0) for v in range(n))
        pend = {u: rules.pending(dist[u], hmin[u], D) for u in range(n) if u not in whole}
        hb = min([x for x in pend.values()] + [NONE])
        if hb == NONE:
            return [d if d != NONE else INF for d in dist]
        for u in [u for u, x in pend.items() if x != NONE and dist[u] < rules.below(hb, min(hmin))]:
            whole.add(u)
            for v in np.flatnonzero(W[u] < INF):
                if v != u:
                    dist[v] = min(dist[v], dist[u] + int(W[u, v]))
    raise AssertionError(f"no end after {rounds} rounds of whole rows")


@pytest.mark.parametrize("wlo,whi", [(0, 0), (0, 1), (0, 3), (1, 1), (1, 4)])
@pytest.mark.parametrize("directed", [False, True])
def test_whole_rows_end(orc, rules, wlo, whi, directed):
    for n, p, cap in ((80, 1.0, 64), (40, 0.8, 3), (33, 0.5, 1), (70, 0.9, 8)):
        rng = np.random.default_rng(n + whi)
        k = rng.random((n, n)) < p
        k = np.triu(k, 1) if not directed else k & ~np.eye(n, dtype=bool)
        src, dst = (x.astype(np.int32) for x in np.nonzero(k))
        w = rng.integers(wlo, whi + 1, src.size).astype(np.int32)
        W = orc.build_matrix(n, src, dst, w, directed)
        for partial in (True, False):
            rows, hmin = build_index(W, cap, partial)
            for s in (0, n - 1):
                assert solve(W, s, rows, hmin, rules) == list(orc.dijkstra(W, s)[0]), (n, cap, partial, s)


def test_trial_is_for_graphs_that_may_take_the_engine(rules):
    assert rules.needs_trial(5, 1) == 1
    assert rules.needs_trial(INF, 1) == 0  # every list complete
    assert rules.needs_trial(5, 0) == 0 and rules.needs_trial(0, 0) == 0  # weights of 0


def test_unaligned_edge_arrays_are_not_read_in_place(rules):
    for a in range(4096, 4104):
        for place in range(3):
            at = [8192, 12288, 16384]
            at[place] = a
            assert rules.in_place(*at) == (a % 4 == 0), at


def test_unaligned_matrix_is_not_read_in_place(rules):
    assert [rules.upload_in_place(4096 + i) for i in range(5)] == [1, 0, 0, 0, 1]


@pytest.mark.parametrize("n", [1, 2, 3, 8, 9, 1000, 262145])
def test_trial_source_has_edges(rules, n):
    """n / 2 if it lists as many edges as any, else a row that does; never a row without edges while one has some."""
    h = n // 2
    best = lambda rows: rules.trial_source(max(rules.trial_word(u, c, e, n) for u, c, e in rows), n)
    nodes = sorted({0, 1 % n, h, n - 1})
    assert best([(u, 64, 1) for u in nodes]) == h
    for u in nodes:
        assert best([(v, 0, int(v == u)) for v in nodes]) == u  # only u has edges (all too heavy to list)
        assert best([(v, 128 if v == u else 127, 1) for v in nodes]) == u
        assert rules.trial_word(u, 128, 1, n) < 2**32


def test_trial_verdict(rules):
    no, every, ask = 0, 1, 2
    assert rules.verdict(0, 0, 0) == no  # did not reach every node that something leads to
    assert rules.verdict(5, 10, 0) == no and rules.verdict(4, 10, 32) == every
    assert rules.verdict(0, 10, 33) == ask
    assert not rules.risky(NONE, 1, 5) and not rules.risky(INF, 1, 5) and not rules.risky(3, INF, 5)
    assert rules.risky(3, 8, 5) and not rules.risky(3, 9, 5)


@pytest.mark.parametrize("cap", [2, 5, 12])
def test_rows_not_at_risk_are_never_pending(orc, rules, cap):
    """Symmetric matrices, random and in parts on a chain or a star: whatever the source, a row pending at the
    end of its solve is one that the trial from any other source counts."""
    rng = np.random.default_rng(cap)
    for trial in range(25):
        n = int(rng.integers(6, 40))
        parts = int(rng.integers(1, 4))
        part = np.arange(n) % parts
        far = int(rng.choice([1, 20, 60]))
        k = np.triu(rng.random((n, n)) < rng.choice([0.3, 0.9]), 1)
        w = rng.integers(1, int(rng.choice([2, 5, 60])) + 1, (n, n)) + far * np.abs(part[:, None] - part[None, :])
        k &= (np.abs(part[:, None] - part[None, :]) <= 1) | (rng.random((n, n)) < 0.1)
        src, dst = (x.astype(np.int32) for x in np.nonzero(k))
        W = orc.build_matrix(n, src, dst, w[src, dst].astype(np.int32), False)
        _, hmin = build_index(W, cap, True)
        dist = [orc.dijkstra(W, s)[0].astype(np.int64) for s in range(n)]
        reached = [d < INF for d in dist]
        if any(not r.all() for r in reached):
            continue
        pending = [{u for u in range(n) if rules.pending(int(d[u]), hmin[u], int(d.max())) != NONE} for d in dist]
        for t in range(n):
            D = int(dist[t].max())
            risk = {u for u in range(n) if rules.risky(int(dist[t][u]), hmin[u], D)}
            for s in range(n):
                assert pending[s] <= risk, (trial, s, t)


def test_few_phases(rules):
    for wmin in (1, 7, 2**30):  # the largest dist is guess - 1
        assert rules.few(2047, min(3 * wmin + 1, 2**31 - 1), wmin) == 1
        assert rules.few(2048, 2, wmin) == 0
    assert rules.few(100, 5, 1) == 0 and rules.few(100, 4, 1) == 1 and rules.few(100, 23, 7) == 0
    assert rules.few(100, 0, 1) == 0  # no trial
