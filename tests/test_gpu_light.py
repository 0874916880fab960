"""The light engine (the default on graphs of positive weights) against the oracle: sizes at the
edges of its lists, slices and key words, rows whose lists are complete, cut or empty, nodes nothing
leads to, and sources for which the lists do not suffice and rows are relaxed whole."""
import time

import numpy as np
import pytest

import graphgen

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dj():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2504_03667_gb300 import dj as _dj
    torch.cuda.set_device(0)
    return _dj


def check(dj, orc, e, sources, what):
    import torch
    W = orc.build_matrix(e.n, e.src, e.dst, e.w, e.directed)
    graphs = [dj.dj_load_edges(e.n, e.src, e.dst, e.w, e.directed),
              dj.dj_load_edges_csr(e.n, e.src, e.dst, e.w, e.directed)]
    k = len(sources)
    D = torch.full((2 * k, e.n), -5, dtype=torch.int32, device="cuda")
    P = torch.full((2 * k, e.n), -5, dtype=torch.int32, device="cuda")
    for j, g in enumerate(graphs):
        for i, s in enumerate(sources):
            dj.dj_sssp(g, s, D[j * k + i], P[j * k + i])
    dj.dj_sync()
    B = torch.full((2, k, e.n), -5, dtype=torch.int32, device="cuda")
    dj.dj_sssp_batch([graphs[0]] * k, sources, list(B[0]), list(B[1]))
    dj.dj_sync()
    for i, s in enumerate(sources):
        ref = orc.dijkstra(W, s)
        got = [("dense", D[i], P[i]), ("compressed rows", D[k + i], P[k + i]), ("batch", B[0, i], B[1, i])]
        for form, d, p in got:
            assert np.array_equal(d.cpu().numpy(), ref[0]), f"{what}, {form}, s={s}: dist"
            assert np.array_equal(p.cpu().numpy(), ref[1]), f"{what}, {form}, s={s}: pred"
    for g in graphs:
        g.free()


@pytest.mark.parametrize("n", [1, 2, 31, 32, 33, 63, 64, 65, 66, 130, 1000, 2047, 2049, 4095, 4097])
def test_sizes(dj, orc, n):
    for wlo, whi, deg, directed in ((1, 3, 4, True), (1, 1000, 70, False), (1, 1, 9, False), (7, 9, 200, True)):
        m = min(n * deg, max(n * (n - 1), 1))
        e = graphgen.random_edges(n, m, wlo, whi, seed=7 * n + deg, directed=directed)
        check(dj, orc, e, sorted({0, n // 2, n - 1}), f"n={n} w in [{wlo}, {whi}] deg {deg}")


def far_source(n, p, seed):
    """A dense directed graph where nothing leads to nodes 0 and n/2, and node 1 is near n/2 but far
    from 0: from n/2 the lists suffice, from 0 every row's unlisted edges stay below the largest
    distance, so every row is relaxed whole."""
    b = graphgen.bernoulli(n, p, 1, 1000, seed)
    h = n // 2
    src, dst, w = np.concatenate([b.src, b.dst]), np.concatenate([b.dst, b.src]), np.concatenate([b.w, b.w])
    keep = (dst != 0) & (dst != h) & (dst != 1)
    src = np.concatenate([src[keep], [h, 0]]).astype(np.int32)
    dst = np.concatenate([dst[keep], [1, 1]]).astype(np.int32)
    w = np.concatenate([w[keep], [1, 3000]]).astype(np.int32)
    return graphgen.EdgeList(n, src, dst, w, True)


@pytest.mark.parametrize("n", [2048, 6143, 6145, 8200])
def test_forms_agree(dj, orc, n):
    """A solve on an idle stream and solves behind one another on a stream may take different forms
    (one cluster, every SM); all are Algorithm 1's, into one buffer pair and into their own."""
    import torch
    for e in (graphgen.bernoulli(n, 0.2, 1, 1000, n), graphgen.outdeg(n, 5, 1, 500, n + 1)):
        W = orc.build_matrix(e.n, e.src, e.dst, e.w, e.directed)
        srcs = [int(x) for x in graphgen.sources(n, 6, 3)]
        refs = [orc.dijkstra(W, s) for s in srcs]
        for load in (dj.dj_load_edges, dj.dj_load_edges_csr):
            g = load(e.n, e.src, e.dst, e.w, e.directed)
            st = torch.cuda.Stream()
            D = torch.full((6, n), -5, dtype=torch.int32, device="cuda")
            P = torch.full((6, n), -5, dtype=torch.int32, device="cuda")
            torch.cuda.synchronize()
            for i, s in enumerate(srcs):  # back to back
                dj.dj_sssp(g, s, D[i], P[i], st)
            dj.dj_sync(st)
            for i in range(6):
                assert np.array_equal(D[i].cpu().numpy(), refs[i][0]) and np.array_equal(P[i].cpu().numpy(), refs[i][1]), i
            for i, s in enumerate(srcs):  # each alone
                dj.dj_sssp(g, s, D[0], P[0], st)
                dj.dj_sync(st)
                assert np.array_equal(D[0].cpu().numpy(), refs[i][0]) and np.array_equal(P[0].cpu().numpy(), refs[i][1]), i
            for s in srcs:  # one buffer pair: the last solve wins
                dj.dj_sssp(g, s, D[0], P[0], st)
            dj.dj_sync(st)
            assert np.array_equal(D[0].cpu().numpy(), refs[5][0]) and np.array_equal(P[0].cpu().numpy(), refs[5][1])
            cg = torch.cuda.CUDAGraph()
            with torch.cuda.graph(cg, stream=st):
                for i, s in enumerate(srcs):
                    dj.dj_sssp(g, s, D[i], P[i], st)
            D.fill_(-5)
            torch.cuda.synchronize()
            cg.replay()
            torch.cuda.synchronize()
            for i in range(6):
                assert np.array_equal(D[i].cpu().numpy(), refs[i][0]) and np.array_equal(P[i].cpu().numpy(), refs[i][1]), i
            del cg
            g.free()


@pytest.mark.parametrize("n", [700, 3001, 4500])
def test_rows_relaxed_whole(dj, orc, n):
    check(dj, orc, far_source(n, 0.4, n), [0, 1, n // 2], f"far source n={n}")


def test_lists_cut_in_ties(dj, orc):
    """Rows with more edges of one weight than the list or its buffer holds, next to light ones."""
    rng = np.random.default_rng(3)
    n = 1500
    src = np.repeat(np.arange(n, dtype=np.int32), 600)
    dst = rng.integers(0, n, src.shape[0]).astype(np.int32)
    w = np.where(rng.random(src.shape[0]) < 0.02, rng.integers(1, 5, src.shape[0]), 40).astype(np.int32)
    check(dj, orc, graphgen.EdgeList(n, src, dst, w, True), [0, 77, n - 1], "weights 1..4 and many 40s")
    check(dj, orc, graphgen.EdgeList(n, src, dst, w, False), [5], "the same undirected")


@pytest.mark.parametrize("n", [130, 400, 1500, 3001, 6143, 6145])
def test_longer_lists(dj, orc, n):
    """About 30 edges per row and unit of weight: lists of 64 edges are too short for most sources, lists of
    128 long enough; then an upload takes the same handle (and a captured solve) back to lists of 64."""
    import torch
    p = min(300 / n, 0.9)
    whi = max(2, round(p * n / 30))
    for directed in (False, True):
        e = (graphgen.random_edges(n, 30 * whi * n, 1, whi, seed=n, directed=True) if directed
             else graphgen.bernoulli(n, p, 1, whi, n))
        check(dj, orc, e, sorted({0, n // 3, n // 2, n - 1}), f"n={n} directed={directed}")
    a, b = graphgen.bernoulli(n, p, 1, whi, n + 1), graphgen.bernoulli(n, p / 2, 1, 40, n + 2)
    st = torch.cuda.Stream()
    d = torch.empty(n, dtype=torch.int32, device="cuda")
    q = torch.empty_like(d)
    G = dj.dj_load_edges(n, a.src, a.dst, a.w, False)
    dj.dj_sssp(G, 5, d, q, st)
    dj.dj_sync(st)
    cg = torch.cuda.CUDAGraph()
    with torch.cuda.graph(cg, stream=st):
        dj.dj_sssp(G, 5, d, q, st)
    W = orc.build_matrix(n, b.src, b.dst, b.w, False)
    ref = orc.dijkstra(W, 5)
    dj.dj_graph_upload(G, W, st)
    d.fill_(-5)
    torch.cuda.synchronize()
    cg.replay()
    torch.cuda.synchronize()
    assert np.array_equal(d.cpu().numpy(), ref[0]) and np.array_equal(q.cpu().numpy(), ref[1])
    del cg
    G.free()


def test_hub_rows(dj, orc):
    """Stars: one row much longer than the others (taken by a whole block in compressed rows)."""
    n = 9001
    rng = np.random.default_rng(4)
    hub = np.zeros(n - 1, dtype=np.int32)
    rim = np.arange(1, n, dtype=np.int32)
    ring = np.stack([rim, np.roll(rim, 1)])
    src = np.concatenate([hub, ring[0]])
    dst = np.concatenate([rim, ring[1]])
    w = np.concatenate([rng.integers(500, 900, n - 1), rng.integers(1, 4, n - 1)]).astype(np.int32)
    check(dj, orc, graphgen.EdgeList(n, src, dst, w, False), [0, 1, 4500], "hub and ring")


def test_upload_rebuilds_the_index(dj, orc):
    """After an upload the same handle (and a captured solve) answers for the new matrix, from aligned
    and unaligned pinned buffers and from pageable memory."""
    import torch
    for n in (203, 4500, 6200):  # the last beyond the CTA form
        a = graphgen.bernoulli(n, 0.3, 1, 1000, 1)
        b = graphgen.bernoulli(n, 0.4, 1, 2, 2)  # the replayed solves need whole rows on it
        Wb = orc.build_matrix(n, b.src, b.dst, b.w, False)
        ref = orc.dijkstra(Wb, 5)
        pinned = torch.from_numpy(Wb).pin_memory()
        padded = torch.empty((n, n + 3), dtype=torch.int32).pin_memory()
        padded[:, 1:n + 1] = pinned
        d = torch.empty(n, dtype=torch.int32, device="cuda")
        p = torch.empty_like(d)
        for what, src in (("pinned", pinned), ("offset", padded[:, 1:n + 1]), ("pageable", Wb)):
            G = dj.dj_load_edges(n, a.src, a.dst, a.w, False)
            st = torch.cuda.Stream()
            dj.dj_sssp(G, 5, d, p, st)
            dj.dj_sync(st)
            cg = torch.cuda.CUDAGraph()
            with torch.cuda.graph(cg, stream=st):
                dj.dj_sssp(G, 5, d, p, st)
            dj.dj_graph_upload(G, src, st)
            d.fill_(-5)
            torch.cuda.synchronize()
            dj.dj_sssp(G, 5, d, p, st)
            dj.dj_sync(st)
            assert np.array_equal(d.cpu().numpy(), ref[0]) and np.array_equal(p.cpu().numpy(), ref[1]), (n, what)
            d.fill_(-5)
            cg.replay()
            torch.cuda.synchronize()
            assert np.array_equal(d.cpu().numpy(), ref[0]) and np.array_equal(p.cpu().numpy(), ref[1]), (n, what, "replay")
            del cg
            G.free()


def test_server_replans(dj, orc):
    """A running server takes a larger graph, then one the light engine does not take, then an upload:
    every request is answered for the graph as it is."""
    import torch
    small, large = graphgen.bernoulli(150, 0.3, 1, 1000, 5), graphgen.bernoulli(3000, 0.05, 1, 1000, 6)
    narrow = graphgen.bernoulli(900, 0.5, 1, 2, 7)
    g = [dj.dj_load_edges(e.n, e.src, e.dst, e.w, False) for e in (small, large, narrow)]
    W = [orc.build_matrix(e.n, e.src, e.dst, e.w, False) for e in (small, large, narrow)]
    srv = dj.dj_serve_create(dj.make_serve_opts(max_slots=8, idle_timeout_ns=300_000_000))

    def ask(gid, k, s):
        t = dj.dj_serve_submit(srv, gid, s)
        assert t is not None
        dj.dj_serve_wait(srv, t)
        got, ref = dj.dj_serve_result(srv, t, W[k].shape[0]), orc.dijkstra(W[k], s)
        assert np.array_equal(got[0], ref[0]) and np.array_equal(got[1], ref[1]), (k, s)

    ids = []
    for k in range(3):  # each added while the kernel planned for the earlier ones is running
        ids.append(dj.dj_serve_add_graph(srv, g[k]))
        for j in range(k + 1):
            ask(ids[j], j, 7 * j + 3)
    srv.destroy()
    srv = dj.dj_serve_create(dj.make_serve_opts(max_slots=8, idle_timeout_ns=300_000_000))
    gid = dj.dj_serve_add_graph(srv, g[1])
    ask(gid, 1, 11)
    W[1] = orc.build_matrix(3000, large.src, large.dst, (large.w % 3 + 1).astype(np.int32), False)
    dj.dj_graph_upload(g[1], torch.from_numpy(W[1]).pin_memory(), torch.cuda.Stream())
    time.sleep(0.05)  # the upload is done; the server still runs
    ask(gid, 1, 12)
    srv.destroy()
    for x in g:
        x.free()


@pytest.mark.parametrize("n,p,whi", [(80, 1.0, 0), (700, 1.0, 0), (700, 0.5, 3), (2049, 0.5, 2), (4097, 0.3, 1)])
def test_many_weights_of_zero(dj, orc, n, p, whi):
    """Rows with more edges of weight 0 than a list holds: loaded, solved and batched as any graph."""
    b = graphgen.bernoulli(n, p, 0, whi, n)
    check(dj, orc, b, [0, n // 2], f"n={n} w in [0, {whi}]")
    e = graphgen.EdgeList(n, np.concatenate([b.src, b.dst]), np.concatenate([b.dst, b.src]),
                          np.concatenate([b.w, np.maximum(b.w, 1)]), True)
    check(dj, orc, e, [n - 1], f"n={n} w in [0, {whi}] directed")


@pytest.mark.parametrize("n,directed", [(400, False), (3001, False), (4500, True)])
def test_captured_solve_ends_on_weights_of_zero(dj, orc, n, directed):
    """A solve captured on positive weights and replayed on a matrix of many zeros ends, with Algorithm 1's dist."""
    import torch
    a = graphgen.bernoulli(n, 0.3, 1, 1000, n)
    b = graphgen.bernoulli(n, 0.6, 0, 2, n + 1)
    W = orc.build_matrix(n, b.src, b.dst, b.w, False)
    st = torch.cuda.Stream()
    d = torch.empty(n, dtype=torch.int32, device="cuda")
    q = torch.empty_like(d)
    both = [np.concatenate(x) for x in ((a.src, a.dst), (a.dst, a.src), (a.w, a.w))]
    G = dj.dj_load_edges(n, *both, True) if directed else dj.dj_load_edges(n, a.src, a.dst, a.w, False)
    dj.dj_sssp(G, 5, d, q, st)
    dj.dj_sync(st)
    cg = torch.cuda.CUDAGraph()
    with torch.cuda.graph(cg, stream=st):
        dj.dj_sssp(G, 5, d, q, st)
    dj.dj_graph_upload(G, W, st)
    torch.cuda.synchronize()
    cg.replay()
    torch.cuda.synchronize()
    assert np.array_equal(d.cpu().numpy(), orc.dijkstra(W, 5)[0])
    del cg
    G.free()


@pytest.mark.parametrize("n", [1500, 3001, 6001])
def test_longer_lists_end_with_an_upload(dj, orc, n):
    """A solve and a batch captured on lists of 128 edges, replayed on another matrix of the same kind: its
    lists are cut at 64, where many rows would go on, and what lay behind them is the old matrix's."""
    import torch
    p = 300 / n
    a, b = graphgen.bernoulli(n, p, 1, 10, n + 1), graphgen.bernoulli(n, p, 1, 10, n + 2)
    W = orc.build_matrix(n, b.src, b.dst, b.w, False)
    srcs = [5, n // 2, n - 1]
    refs = [orc.dijkstra(W, s) for s in srcs]
    pinned = torch.from_numpy(W).pin_memory()
    padded = torch.empty((n, n + 3), dtype=torch.int32).pin_memory()
    padded[:, 1:n + 1] = pinned
    for what, src in (("pageable", W), ("pinned", pinned), ("offset", padded[:, 1:n + 1])):
        st = torch.cuda.Stream()
        D = torch.empty((2, 3, n), dtype=torch.int32, device="cuda")
        P = torch.empty_like(D)
        G = dj.dj_load_edges(n, a.src, a.dst, a.w, False)
        batch = dj.dj_batch_create([G] * 3, srcs, list(D[1]), list(P[1]))

        def solve():
            for i, s in enumerate(srcs):
                dj.dj_sssp(G, s, D[0, i], P[0, i], st)
            dj.dj_batch_launch(batch, st)

        solve()
        dj.dj_sync(st)
        cg = torch.cuda.CUDAGraph()
        with torch.cuda.graph(cg, stream=st):
            solve()
        dj.dj_graph_upload(G, src, st)
        for how, again in (("replay", cg.replay), ("new calls", solve)):
            torch.cuda.synchronize()
            D.fill_(-5)
            P.fill_(-5)
            torch.cuda.synchronize()
            again()
            torch.cuda.synchronize()
            for j, form in enumerate(("single", "batch")):
                for i in range(3):
                    assert np.array_equal(D[j, i].cpu().numpy(), refs[i][0]), (what, how, form, i)
                    assert np.array_equal(P[j, i].cpu().numpy(), refs[i][1]), (what, how, form, i)
        del cg
        batch.free()
        G.free()


def without(e, nodes):
    """e with the given nodes isolated."""
    keep = ~(np.isin(e.src, nodes) | np.isin(e.dst, nodes))
    return graphgen.EdgeList(e.n, e.src[keep], e.dst[keep], e.w[keep], e.directed)


def star(parts, size, bridge, seed):
    """Dense parts whose first nodes hang on the middle part's: from that node the lists suffice."""
    es = [graphgen.bernoulli(size, 0.5, 1, 1000, seed + i) for i in range(parts)]
    hubs = np.arange(parts, dtype=np.int32) * size
    mid = hubs[parts // 2]
    src = np.concatenate([e.src + h for e, h in zip(es, hubs)] + [np.full(parts - 1, mid)])
    dst = np.concatenate([e.dst + h for e, h in zip(es, hubs)] + [hubs[hubs != mid]])
    w = np.concatenate([e.w for e in es] + [np.full(parts - 1, bridge)])
    return graphgen.EdgeList(parts * size, src.astype(np.int32), dst.astype(np.int32), w.astype(np.int32), False)


@pytest.mark.parametrize("n", [300, 1500, 5000])
def test_one_source_says_nothing_about_the_others(dj, orc, n):
    """Graphs whose middle node leads nowhere, into a small part, or is nearer to everything than any other."""
    h = n // 2
    for whi in (2, 10, 1000):
        b = graphgen.bernoulli(n, 0.4, 1, whi, n)
        check(dj, orc, without(b, [h]), [0, h, n - 1], f"n={n} isolated middle, w up to {whi}")
    d = graphgen.EdgeList(n, np.concatenate([b.src, b.dst]), np.concatenate([b.dst, b.src]),
                          np.concatenate([b.w, b.w]), True)
    keep = d.src != h
    check(dj, orc, graphgen.EdgeList(n, d.src[keep], d.dst[keep], d.w[keep], True), [1, h], f"n={n} sink in the middle")
    two = without(b, [h, h + 1])
    keep = (two.src < h) == (two.dst < h)
    pair = graphgen.EdgeList(n, np.append(two.src[keep], h).astype(np.int32), np.append(two.dst[keep], h + 1).astype(np.int32),
                             np.append(two.w[keep], 7).astype(np.int32), False)
    check(dj, orc, pair, [0, h, n - 1], f"n={n} two parts and a pair")
    for bridge in (20, 150):
        check(dj, orc, star(3, n // 3, bridge, n), [0, n // 3 + 5, n // 3 * 3 - 1], f"n={n} star, bridge {bridge}")


@pytest.mark.parametrize("n", [70, 300, 599, 600, 1500, 2047, 2048])
def test_few_phases(dj, orc, n):
    """Narrow weights: a largest dist of two or three, lists of 64 cut, alone, behind others and batched; and a
    batch with another graph."""
    import torch
    for p, whi in ((min(0.95, 250 / n), 1), (min(0.95, 250 / n), 3), (min(0.95, 400 / n), 9)):
        e = graphgen.bernoulli(n, p, 1, whi, n)
        check(dj, orc, e, sorted({0, n // 2, n - 1}), f"n={n} p={p:.2f} w up to {whi}")
    b = graphgen.bernoulli(900, 0.3, 1, 1000, n)
    gs = [dj.dj_load_edges(x.n, x.src, x.dst, x.w, False) for x in (e, b)]
    outs = [[torch.empty(x.n, dtype=torch.int32, device="cuda") for x in (e, b)] for _ in range(2)]
    dj.dj_sssp_batch(gs, [1, 1], outs[0], outs[1])
    dj.dj_sync()
    for i, x in enumerate((e, b)):
        ref = orc.dijkstra(orc.build_matrix(x.n, x.src, x.dst, x.w, False), 1)
        assert np.array_equal(outs[0][i].cpu().numpy(), ref[0]) and np.array_equal(outs[1][i].cpu().numpy(), ref[1]), i
    for g in gs:
        g.free()


@pytest.mark.parametrize("n,p", [(70, 0.95), (1024, 0.3), (2500, 0.1), (3000, 0.3)])
def test_directed_matrices_with_cut_lists(dj, orc, n, p):
    """Alone, behind one another, captured and after an upload: the answer is the same whichever engine takes them."""
    import torch
    b = [graphgen.bernoulli(n, p, 1, 1000, n + i) for i in range(2)]
    e = graphgen.EdgeList(n, np.concatenate([b[0].src, b[1].dst]), np.concatenate([b[0].dst, b[1].src]),
                          np.concatenate([b[0].w, b[1].w]), True)
    W = orc.build_matrix(n, e.src, e.dst, e.w, True)
    srcs = [0, n // 2, n - 1]
    refs = [orc.dijkstra(W, s) for s in srcs]
    for g in (dj.dj_load_edges(n, e.src, e.dst, e.w, True), dj.dj_load_dense(W)):
        st = torch.cuda.Stream()
        D = torch.empty((3, n), dtype=torch.int32, device="cuda")
        P = torch.empty_like(D)

        def solve(alone):
            for i, s in enumerate(srcs):
                dj.dj_sssp(g, s, D[i], P[i], st)
                if alone:
                    dj.dj_sync(st)

        solve(True)
        cg = torch.cuda.CUDAGraph()
        with torch.cuda.graph(cg, stream=st):
            solve(False)
        for how, again in (("alone", lambda: solve(True)), ("behind", lambda: solve(False)), ("captured", cg.replay),
                           ("uploaded", lambda: (dj.dj_graph_upload(g, W, st), solve(False)))):
            torch.cuda.synchronize()
            D.fill_(-5)
            P.fill_(-5)
            torch.cuda.synchronize()
            again()
            torch.cuda.synchronize()
            for i in range(3):
                assert np.array_equal(D[i].cpu().numpy(), refs[i][0]), (how, i)
                assert np.array_equal(P[i].cpu().numpy(), refs[i][1]), (how, i)
        del cg
        g.free()


@pytest.mark.parametrize("kind", ["large", "longer lists", "few phases", "directed"])
def test_solves_on_many_streams(dj, orc, kind):
    """More streams than the library keeps a word for, several solves on each, some behind an event, a copy or
    another kernel, some captured (alone and behind one another): every form gives the same answer."""
    import torch
    n = 6200 if kind == "large" else 1500
    if kind == "directed":
        b = graphgen.bernoulli(n, 0.2, 1, 1000, 1)
        e = graphgen.EdgeList(n, np.concatenate([b.src, b.dst]), np.concatenate([b.dst, b.src]),
                              np.concatenate([b.w, b.w[::-1]]), True)
    else:
        p, whi = {"large": (0.05, 1000), "longer lists": (0.2, 10), "few phases": (0.5, 9)}[kind]
        e = graphgen.bernoulli(n, p, 1, whi, 1)
    W = orc.build_matrix(n, e.src, e.dst, e.w, e.directed)
    srcs = [0, 7, n - 1]
    refs = [orc.dijkstra(W, s) for s in srcs]
    g = dj.dj_load_edges(n, e.src, e.dst, e.w, e.directed)
    streams = [torch.cuda.Stream() for _ in range(70)]
    D = torch.empty((len(streams), 3, n), dtype=torch.int32, device="cuda")
    P = torch.empty_like(D)

    def run(j):
        for i, s in enumerate(srcs):
            with torch.cuda.stream(streams[j]):
                if (i + j) % 4 == 1:
                    torch.cuda.Event().record()
                elif (i + j) % 4 == 2:
                    D[j, i].fill_(-9)
            dj.dj_sssp(g, s, D[j, i], P[j, i], streams[j])

    graphs = []
    run(0)
    torch.cuda.synchronize()
    for j in (0, 1):  # one solve a graph, and three
        cg = torch.cuda.CUDAGraph()
        with torch.cuda.graph(cg, stream=streams[j]):
            for i in range(1 if j == 0 else 3):
                dj.dj_sssp(g, srcs[i], D[j, i], P[j, i], streams[j])
        graphs.append(cg)
    for turn in range(3):
        D.fill_(-5)
        P.fill_(-5)
        torch.cuda.synchronize()
        for j in range(len(streams)):
            if turn == 2 and j < 2:
                graphs[j].replay()
            else:
                run(j)
        torch.cuda.synchronize()
        d, p = D.cpu().numpy(), P.cpu().numpy()
        for j in range(len(streams)):
            for i in range(1 if turn == 2 and j == 0 else 3):
                assert np.array_equal(d[j, i], refs[i][0]) and np.array_equal(p[j, i], refs[i][1]), (turn, j, i)
    del graphs
    g.free()
