"""The work a user of this library has it do, as cases that can be timed and compared.

Every case goes through the public binding (paper_2504_03667_gb300.dj): graphs are loaded from
host edge lists as a program does, and a pass is one call (or the few calls) such a program makes
with the graph in hand.  Inputs are seeded; shapes, densities and weight ranges are those of the
workloads in graphgen, of the tests and of bench.py, with ragged sizes between them.

Kinds:
  single  dj_sssp on a resident matrix (n, density p or out-degree d, weight range)
  csr     dj_sssp on a graph loaded in compressed-row form
  batch   a prepared batch: k sources of one graph in one launch
  mixed   dj_sssp_batch, one call, on graphs of different sizes
  serve   dj_serve on resident graphs, every request waiting at the start
  load    edge list in host memory -> graph -> one solve -> host results
  upload  a new matrix in pinned host memory -> dj_graph_upload -> one solve -> host results
"""
import math

import numpy as np
import torch

from paper_2504_03667_gb300 import dj


def listed():
    return [
        # the smallest call: a small directed network, one route query; launch latency counts
        {"name": "single_n200_d6", "kind": "single", "n": 200, "d": 6, "wlo": 1, "whi": 100},
        # the plain single-source workload of a small dense graph
        {"name": "single_n1024_p0.1", "kind": "single", "n": 1024, "p": 0.1, "wlo": 1, "whi": 100},
        # an ordinary dense graph of odd size
        {"name": "single_n5003_p0.3", "kind": "single", "n": 5003, "p": 0.3, "wlo": 1, "whi": 1000},
        # few distinct weights: almost every path has ties to break
        {"name": "single_n6001_ties", "kind": "single", "n": 6001, "p": 0.05, "wlo": 1, "whi": 10},
        # the headline: a dense graph whose matrix is 1 GiB
        {"name": "single_n16384_p0.5", "kind": "single", "n": 16384, "p": 0.5, "wlo": 1, "whi": 1000},
        # a sparse directed graph stored densely, a 4 GiB matrix (the largest resident graph)
        {"name": "single_n32768_d8", "kind": "single", "n": 32768, "d": 8, "wlo": 1, "whi": 10000},
        # the same graph without the matrix
        {"name": "csr_n32768_d8", "kind": "csr", "n": 32768, "d": 8, "wlo": 1, "whi": 10000},
        # many sources of one graph (all-pairs blocks, centralities): throughput
        {"name": "batch_n8192_k256", "kind": "batch", "n": 8192, "p": 0.05, "wlo": 1, "whi": 1000, "k": 256},
        # one call over a collection of graphs of uneven size
        {"name": "mixed_48_graphs", "kind": "mixed", "graphs": 48, "nlo": 100, "nhi": 4000, "plo": 0.02, "phi": 0.5,
         "wlo": 1, "whi": 1000},
        # a server under a burst of requests
        {"name": "serve_24g_1500r", "kind": "serve", "graphs": 24, "requests": 1500, "nlo": 512, "nhi": 8192,
         "plo": 0.01, "phi": 0.5, "wlo": 1, "whi": 1000},
        # one-off use: build the graph from an edge list, solve once, read the answer
        {"name": "load_n4099_p0.3", "kind": "load", "n": 4099, "p": 0.3, "wlo": 1, "whi": 1000},
        # a matrix that changes between solves: upload, solve, read the answer
        {"name": "upload_n8192_p0.5", "kind": "upload", "n": 8192, "p": 0.5, "wlo": 1, "whi": 1000},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _weights(rng):
    return rng.choice([(1, 100), (1, 1000), (1, 1000), (1, 10000), (1, 10), (0, 100)])


def draw(rng):
    kind = rng.choice(["single", "single", "single", "single", "csr", "csr", "batch", "batch", "mixed", "serve", "load",
                       "upload"])
    wlo, whi = _weights(rng)
    c = {"kind": kind, "wlo": wlo, "whi": whi}
    if kind == "single":
        if rng.random() < 0.35:
            c.update(n=_log(rng, 100, 32768), d=rng.randint(3, 16))
        else:
            c.update(n=_log(rng, 64, 16384), p=round(math.exp(rng.uniform(math.log(0.02), math.log(0.5))), 4))
    elif kind == "csr":
        c.update(n=_log(rng, 500, 100000), d=rng.randint(3, 16))
    elif kind == "batch":
        c.update(n=_log(rng, 200, 8192), p=round(math.exp(rng.uniform(math.log(0.02), math.log(0.3))), 4),
                 k=_log(rng, 8, 256), wlo=max(wlo, 1))
    elif kind == "mixed":
        c.update(graphs=rng.randint(4, 48), nlo=rng.randint(40, 400), nhi=rng.randint(1000, 4000), plo=0.02, phi=0.5,
                 wlo=max(wlo, 1))
    elif kind == "serve":
        c.update(graphs=rng.randint(4, 24), requests=_log(rng, 150, 1500), nlo=rng.randint(100, 600),
                 nhi=rng.randint(2000, 8192), plo=0.01, phi=0.5, wlo=max(wlo, 1))
    elif kind == "load":
        c.update(n=_log(rng, 100, 4099), p=round(rng.uniform(0.02, 0.3), 4))
    else:
        c.update(n=_log(rng, 500, 8192), p=round(rng.uniform(0.02, 0.5), 4), wlo=max(wlo, 1))
    return c


# ---------------------------------------------------------------------- inputs

def _bernoulli(n, p, wlo, whi, gen):
    """Undirected: each pair i < j is an edge with probability p (device tensors src, dst, w)."""
    i = torch.nonzero(torch.rand((n, n), generator=gen, device="cuda").lt_(p).triu_(1) > 0)
    src, dst = i[:, 0].int(), i[:, 1].int()
    w = torch.randint(wlo, whi + 1, (src.numel(),), generator=gen, device="cuda", dtype=torch.int32)
    return src, dst, w


def _outdeg(n, d, wlo, whi, gen):
    """Directed: d uniform targets per node, repeats kept, self-loops dropped."""
    src = torch.arange(n, device="cuda", dtype=torch.int32).repeat_interleave(d)
    dst = torch.randint(0, n, (n * d,), generator=gen, device="cuda", dtype=torch.int32)
    w = torch.randint(wlo, whi + 1, (n * d,), generator=gen, device="cuda", dtype=torch.int32)
    keep = src != dst
    return src[keep], dst[keep], w[keep]


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _edges(case, gen):
    """(n, src, dst, w, directed) of the case's graph, on the device."""
    if "d" in case:
        return (case["n"],) + _outdeg(case["n"], case["d"], case["wlo"], case["whi"], gen) + (True,)
    return (case["n"],) + _bernoulli(case["n"], case["p"], case["wlo"], case["whi"], gen) + (False,)


def _host(e):
    return e[0], e[1].cpu().numpy(), e[2].cpu().numpy(), e[3].cpu().numpy(), e[4]


def _collection(case):
    """The shapes (n, p) of a collection of graphs: n spread evenly over the logarithm of its range
    and p evenly over its own, in orders that have nothing to do with one another."""
    lo, hi = case["nlo"], case["nhi"]
    spread = [((i * 0.6180339887498949) % 1.0, (i * 0.7548776662466927 + 0.5) % 1.0) for i in range(case["graphs"])]
    return [(int(lo * (hi / lo) ** a), case["plo"] + (case["phi"] - case["plo"]) * b) for a, b in spread]


def _all_edges(case, seed):
    """Every graph of the case, the sources, and for a collection the graph of each source."""
    gen = _gen(seed)
    kind = case["kind"]
    if kind in ("mixed", "serve"):
        graphs = [(n,) + _bernoulli(n, p, case["wlo"], case["whi"], gen) + (False,) for n, p in _collection(case)]
        k = case["requests"] if kind == "serve" else len(graphs)
        which = [(7 * i) % len(graphs) for i in range(k)] if kind == "serve" else list(range(k))
        u = torch.rand(k, generator=gen, device="cuda", dtype=torch.float64).tolist()
        return graphs, [int(x * graphs[g][0]) for x, g in zip(u, which)], which
    e = _edges(case, gen)
    k = case.get("k", 1)
    srcs = torch.randperm(case["n"], generator=gen, device="cuda")[:k].tolist()
    return [e], srcs, [0] * len(srcs)


def _rows(sizes):
    """One result buffer and a view of it for each solve."""
    buf = torch.empty(sum(sizes), dtype=torch.int32, device="cuda")
    return buf, list(buf.split(sizes))


def prepare(case, seed):
    kind = case["kind"]
    graphs, srcs, which = _all_edges(case, seed)
    host = [_host(e) for e in graphs]
    sizes = [e[0] for e in graphs]
    del graphs
    if kind == "load":
        return {"kind": kind, "edges": host[0], "source": srcs[0]}
    load = dj.dj_load_edges_csr if kind == "csr" else dj.dj_load_edges
    st = {"kind": kind, "graphs": [load(*h) for h in host], "sources": srcs, "which": which}
    if kind == "upload":
        n = sizes[0]
        st["matrix"] = torch.from_numpy(dj.dj_graph_download(st["graphs"][0])).pin_memory()
        st["host"] = [torch.empty(n, dtype=torch.int32).pin_memory() for _ in range(2)]
        # the program's graph so far holds another matrix of the same size
        old = _host(_edges(case, _gen(seed + 1000003)))
        st["graphs"] = [load(*old)]
        return st
    st["all_dist"], st["dist"] = _rows([sizes[g] for g in which])
    st["all_pred"], st["pred"] = _rows([sizes[g] for g in which])
    if kind == "batch":
        st["batch"] = dj.dj_batch_create([st["graphs"][0]] * len(srcs), srcs, st["dist"], st["pred"])
    elif kind == "serve":
        st["opts"] = dj.make_serve_opts(max_slots=512)
        st["arrival"] = np.zeros(len(srcs))
    return st


def run(state):
    kind = state["kind"]
    if kind in ("single", "csr"):
        dj.dj_sssp(state["graphs"][0], state["sources"][0], state["dist"][0], state["pred"][0])
    elif kind == "batch":
        dj.dj_batch_launch(state["batch"])
    elif kind == "mixed":
        dj.dj_sssp_batch(state["graphs"], state["sources"], state["dist"], state["pred"])
    elif kind == "serve":
        dj.dj_serve(state["graphs"], state["which"], state["sources"], state["arrival"], state["dist"], state["pred"],
                    state["opts"])
    elif kind == "load":
        n, src, dst, w, directed = state["edges"]
        g = dj.dj_load_edges(n, src, dst, w, directed)
        out = dj.dj_sssp_host(g, state["source"])
        g.free()
        return list(out)
    else:
        dj.dj_graph_upload(state["graphs"][0], state["matrix"])
        return list(dj.dj_sssp_host(state["graphs"][0], state["sources"][0], *state["host"]))
    return [state["all_dist"], state["all_pred"]]


# ---------------------------------------------------------------------- what a pass cannot do without

def _arcs(n, case, p=None):
    return n * case["d"] if "d" in case else (case["p"] if p is None else p) * n * n


def work(case):
    kind = case["kind"]
    if kind in ("mixed", "serve"):  # the expected sizes of the collection
        lo, hi, p = case["nlo"], case["nhi"], 0.5 * (case["plo"] + case["phi"])
        n1 = (hi - lo) / math.log(hi / lo)
        n2 = (hi * hi - lo * lo) / (2 * math.log(hi / lo))
        k = case["requests"] if kind == "serve" else case["graphs"]
        return {"bytes": case["graphs"] * n2 * 4 + k * n1 * 8, "flops": 2 * k * p * n2}
    n, k = case["n"], case.get("k", 1)
    arcs = _arcs(n, case)
    if kind == "csr":
        return {"bytes": 8 * arcs + 8 * n + 8 * n, "flops": 2 * arcs}
    if kind == "load":
        return {"bytes": 6 * arcs + 4 * n * n + 8 * n, "flops": 2 * arcs}
    if kind == "upload":
        return {"bytes": 2 * 4 * n * n + 8 * n, "flops": 2 * arcs}
    return {"bytes": 4 * n * n + 8 * n * k, "flops": 2 * k * arcs}


# ---------------------------------------------------------------------- the answer in 64 bits

def _by_rounds(n, src, dst, w, sources):
    """dist by repeated relaxation of every arc; pred[v] is the u of smallest (dist[u], u) among
    those offering dist[v], which is the one Algorithm 1 keeps when every weight is positive."""
    inf = 2 ** 31 - 1
    out = []
    for s in sources:
        d = torch.full((n,), inf, dtype=torch.int64, device="cuda")
        d[s] = 0
        while True:
            x = torch.clamp(d[src] + w, max=inf)
            nd = d.scatter_reduce(0, dst, x, "amin")
            if torch.equal(nd, d):
                break
            d = nd
        tight = (d[src] + w == d[dst]) & (d[src] < inf)
        key = torch.full((n,), 2 ** 62, dtype=torch.int64, device="cuda")
        u = src[tight]
        key.scatter_reduce_(0, dst[tight], d[u] * n + u, "amin")
        p = torch.where(key < 2 ** 62, key % n, torch.full_like(key, -1))
        p[s] = -1
        out.append((d, p))
    return out


def _by_steps(n, src, dst, w, s):
    """Algorithm 1 step by step (zero weights allowed)."""
    inf = 2 ** 31 - 1
    G = np.full((n, n), inf, dtype=np.int64)
    np.minimum.at(G, (src, dst), w)
    np.fill_diagonal(G, inf)
    d = np.full(n, inf, dtype=np.int64)
    open_d = d.copy()
    p = np.full(n, -1, dtype=np.int64)
    d[s] = open_d[s] = 0
    done = np.zeros(n, dtype=bool)
    for _ in range(n):
        u = int(np.argmin(open_d))
        if open_d[u] >= inf:
            break
        done[u] = True
        open_d[u] = inf
        x = d[u] + G[u]
        better = (x < d) & (G[u] < inf) & ~done
        d[better] = x[better]
        open_d[better] = x[better]
        p[better] = u
    return torch.from_numpy(d), torch.from_numpy(p)


def exact(case, seed):
    """None for the server: over a thousand solves.  None for zero weights on large graphs: only
    Algorithm 1's own steps give their pred."""
    if case["kind"] == "serve" or (case["wlo"] == 0 and case["n"] > 8192):
        return None
    graphs, srcs, which = _all_edges(case, seed)
    arcs = []
    for n, a, b, w, directed in graphs:
        if not directed:
            a, b, w = torch.cat([a, b]), torch.cat([b, a]), torch.cat([w, w])
        arcs.append((n, a.long(), b.long(), w.long()))
    if case["wlo"] == 0:
        n, a, b, w = arcs[0]
        res = [_by_steps(n, a.cpu().numpy(), b.cpu().numpy(), w.cpu().numpy(), srcs[0])]
    else:
        res = [r for s, g in zip(srcs, which) for r in _by_rounds(*arcs[g], [s])]
    return [torch.cat([d for d, _ in res]), torch.cat([p for _, p in res])]
