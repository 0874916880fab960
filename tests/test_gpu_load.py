"""Building the matrix from an edge list read by the device itself: every size around the scatter's
grid, arrays at odd offsets, and the first bad edge named whatever its place in the list."""
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


@pytest.mark.parametrize("m", [0, 1, 3, 255, 256, 1023, 1025, 40000])
@pytest.mark.parametrize("directed", [False, True])
def test_matrix_matches_the_fill_rules(dj, orc, m, directed):
    n = 61
    e = graphgen.random_edges(n, m + 1, 0, 9, seed=500 + m, directed=directed)
    src, dst, w = e.src[1:], e.dst[1:], e.w[1:]  # one entry off the arrays' alignment
    G = dj.dj_load_edges(n, src, dst, w, directed)
    assert np.array_equal(dj.dj_graph_download(G), orc.build_matrix(n, src, dst, w, directed))
    G.free()


@pytest.mark.parametrize("at", [0, 1, 1024, 77777, 99999])
def test_first_bad_edge_is_named(dj, at):
    n, m = 500, 100000
    e = graphgen.random_edges(n, m, 1, 9, seed=9, directed=True)
    for what, value, word in (("src", n, "node id"), ("dst", -1, "node id"), ("w", -5, "weight"), ("w", 2**31 - 1, "weight")):
        a = {"src": e.src.copy(), "dst": e.dst.copy(), "w": e.w.copy()}
        a[what][at] = value
        a["w"][min(m - 1, at + 5000)] = -1  # a later one
        with pytest.raises(dj.DjError) as ei:
            dj.dj_load_edges(n, a["src"], a["dst"], a["w"], True)
        assert ei.value.status == dj.DJ_EINVAL
        assert f"edge {at} " in str(ei.value) and word in str(ei.value)
    w = e.w.copy()
    w[at] = (2**31 - 1) // (n - 1) + 1
    if e.src[at] != e.dst[at]:
        with pytest.raises(dj.DjError) as ei:
            dj.dj_load_edges(n, e.src, e.dst, w, True)
        assert ei.value.status == dj.DJ_EOVERFLOW


@pytest.mark.parametrize("n", [1, 3, 31, 33, 130, 517])
def test_dense_matrix_from_aligned_and_odd_places(dj, orc, n):
    """A device matrix at any alignment, and a host one, give the same graph; a negative entry anywhere
    is refused."""
    import torch
    e = graphgen.random_edges(n, 9 * n, 1, 50, seed=n, directed=True)
    W = orc.build_matrix(n, e.src, e.dst, e.w, True)
    room = torch.full((n * n + 8,), -9, dtype=torch.int32, device="cuda")
    for c in (0, 1, 4):
        A = room[c:c + n * n].view(n, n)
        A.copy_(torch.from_numpy(W))
        G = dj.dj_load_dense(A)
        assert np.array_equal(dj.dj_graph_download(G), W)
        d = torch.empty(n, dtype=torch.int32, device="cuda")
        p = torch.empty_like(d)
        dj.dj_sssp(G, n // 2, d, p)
        dj.dj_sync()
        ref = orc.dijkstra(W, n // 2)
        assert np.array_equal(d.cpu().numpy(), ref[0]) and np.array_equal(p.cpu().numpy(), ref[1])
        G.free()
        for r, k in ((0, n - 1), (n - 1, 0)):
            A[r, k] = -1
            with pytest.raises(dj.DjError):
                dj.dj_load_dense(A)
            A[r, k] = int(W[r, k])
        room.fill_(-9)
    G = dj.dj_load_dense(W)
    assert np.array_equal(dj.dj_graph_download(G), W)
    G.free()


@pytest.mark.parametrize("off", [1, 2, 3])
def test_arrays_at_odd_byte_addresses(dj, orc, off):
    """Edge arrays that are not 4-byte aligned (views into a byte buffer) load like any others."""
    n, m = 300, 20000
    e = graphgen.random_edges(n, m, 1, 90, seed=off, directed=True)

    def odd(a):
        buf = bytearray(4 * a.size + 4)
        x = np.frombuffer(buf, np.int32, a.size, off)
        x[:] = a
        assert x.ctypes.data % 4 == off % 4
        return x

    for load in (dj.dj_load_edges, dj.dj_load_edges_csr):
        for odd_src, odd_dst, odd_w in ((1, 1, 1), (1, 0, 0), (0, 1, 0), (0, 0, 1)):
            s, t, w = (odd(a) if o else a for o, a in ((odd_src, e.src), (odd_dst, e.dst), (odd_w, e.w)))
            G = load(n, s, t, w, True)
            if load is dj.dj_load_edges:
                assert np.array_equal(dj.dj_graph_download(G), orc.build_matrix(n, e.src, e.dst, e.w, True))
            G.free()
            bad = e.w.copy()
            bad[m - 3] = -7
            with pytest.raises(dj.DjError) as ei:
                load(n, s, t, odd(bad), True)
            assert f"edge {m - 3} " in str(ei.value) and "weight" in str(ei.value)


@pytest.mark.parametrize("n", [33, 64, 300])
def test_upload_from_an_odd_byte_address(dj, orc, n):
    """A matrix in pinned memory that is not 4-byte aligned uploads like any other."""
    import torch
    e = graphgen.random_edges(n, 9 * n, 1, 90, seed=n, directed=True)
    W = orc.build_matrix(n, e.src, e.dst, e.w, True)
    ref = orc.dijkstra(W, n // 2)
    pinned = torch.zeros(4 * n * n + 4, dtype=torch.uint8).pin_memory()
    for off in (1, 2, 3):
        A = np.frombuffer(pinned.numpy(), np.int32, n * n, off).reshape(n, n)
        A[:] = W
        assert A.ctypes.data % 4 == off
        G = dj.dj_load_edges(n, e.src, e.dst, np.ones(9 * n, np.int32), True)
        dj.dj_graph_upload(G, A)
        got = dj.dj_sssp_host(G, n // 2)
        assert np.array_equal(dj.dj_graph_download(G), W)
        assert np.array_equal(got[0], ref[0]) and np.array_equal(got[1], ref[1])
        G.free()
