"""GPU parity of the frontier engine where its paths hand over to each other.

Each graph drives one branch (an edge with more followers than a block takes,
long windows, few lanes of scratch, no scratch at all); results must equal the
oracle's or another engine's bit for bit.
"""
import numpy as np
import pytest

import oracle
from paper_2010_08423_gb300 import capi
from paper_2010_08423_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    capi.load()
    oracle.build()
    torch.cuda.set_device(0)


def graph_of(src, dst, t, delta, ncolors=0):
    src, dst, t, delta = (np.asarray(x, dtype=np.uint32) for x in (src, dst, t, delta))
    g = {"n": len(delta), "src": src, "dst": dst, "t": t, "delta": delta}
    if ncolors:
        g["color"] = (np.arange(len(delta)) % ncolors).astype(np.uint8)
    return g


def batch(G, n, qs):
    import torch
    nq = len(qs)
    d_w = torch.full((nq, n), -1, dtype=torch.int64, device="cuda")
    d_b = torch.full((nq, (n + 7) // 8), 255, dtype=torch.uint8, device="cuda")
    d_s = torch.full((nq,), -1, dtype=torch.int32, device="cuda")
    capi.rr_reach_batch_device(G.handle, qs, d_w, d_b, d_s)
    torch.cuda.synchronize()
    return d_w.cpu().numpy().view(np.uint64), d_b.cpu().numpy(), d_s.cpu().numpy()


@pytest.mark.parametrize("followers", [1024, 1025, 1500, 40_000])
@pytest.mark.parametrize("edges", [1, 3, 40])
def test_a_source_edge_into_a_hub(followers, edges):
    # layer 1 has few rows, one of which more than 1,024 edges may follow: the
    # query is given up in layer 2, by all warps together (k = 2: after layer 1)
    hub, mid = 1, 2 + np.arange(edges - 1)
    out = 1 + edges + np.arange(followers)
    end = int(out[-1]) + 1
    src = np.concatenate([np.zeros(edges, int), np.full(followers, hub), out, mid])
    dst = np.concatenate([[hub], mid, out, np.full(followers, end), np.full(edges - 1, hub)])
    t = np.concatenate([np.full(edges, 1), np.full(followers, 2), np.full(followers, 3), np.full(edges - 1, 2)])
    g = graph_of(src, dst, t, np.full(end + 1, 2))
    qs = [{"source": 0, "k": 2 + i % 4, "seed": 7 + i, "motif": None} for i in range(300)]
    with capi.Graph(g) as G:
        for q in qs[:4]:
            ref = oracle.sieve(g, 0, q["k"], q["seed"])
            for _ in range(20):
                _, w = G.reach(0, q["k"], q["seed"])
                assert np.array_equal(w, ref), q
            assert w.any() or (q["k"] == 5 and edges == 1)
        w, bm, st = batch(G, g["n"], qs)
        assert not st.any()
        for i, q in enumerate(qs):
            b1, w1 = G.reach(0, q["k"], q["seed"])
            assert np.array_equal(w[i], w1) and np.array_equal(bm[i], b1), i


def exchange(d, wait, ncolors=0, seed=0):
    """A hub 0 and d leaves, an edge from and to every leaf; leaf 1 is the source."""
    rng = np.random.default_rng([seed, d])
    leaf = 1 + np.arange(d)
    tau = 1000
    t = np.concatenate([rng.integers(1, tau, d), rng.integers(1, tau, d)])
    t[0] = tau // 8  # the source's only edge: rows before it have windows without a walk
    delta = np.concatenate([[wait], rng.integers(0, tau, d)])
    src, dst = np.concatenate([leaf, np.zeros(d, int)]), np.concatenate([np.zeros(d, int), leaf])
    return graph_of(src, dst, t, delta, ncolors)


@pytest.mark.parametrize("d,wait", [(4_000, 1000), (16_000, 1000), (17_000, 1000), (23_000, 800),
                                    (150_001, 900), (4_600_000, 1000)])
def test_windows_longer_than_the_direct_reads(d, wait):
    # one dominant vertex and long waits: windows of d rows, by each level of
    # their summaries (from 16,385, 131,000 and 4,194,000 rows on). A second hub
    # continues the paths: leaf, hub, leaf, hub, leaf, and no longer ones (walks
    # of six vertices exist, and cancel)
    import torch
    g = exchange(d, wait, ncolors=2)
    h2 = g["n"]
    rng = np.random.default_rng(d)
    leaf = 1 + np.arange(d)
    g = graph_of(np.concatenate([g["src"], leaf, np.full(d, h2)]), np.concatenate([g["dst"], np.full(d, h2), leaf]),
                 np.concatenate([g["t"], rng.integers(1, 1000, 2 * d)]), np.concatenate([g["delta"], [wait]]), 2)
    n = g["n"]
    ks = (3, 4, 5, 6) if d < 1_000_000 else (5,)
    with capi.Graph(g) as G, capi.Graph(g, capi.FLAG_DENSE_STATE) as H:
        for k in ks:
            for m in (None, [0, 1] * (k // 2) + [1] * (k % 2)):
                b, w = G.reach(1, k, 3 + k, motif=m)
                b1, w1 = H.reach(1, k, 3 + k, motif=m)
                assert np.array_equal(w, w1) and np.array_equal(b, b1), (k, m)
                assert m is not None or w.any() == (k <= 5), k
        if d < 1_000_000:
            d_w = torch.full((4, n), -1, dtype=torch.int64, device="cuda")
            capi.rr_reach_atmost_device(G.handle, 1, 5, 9, d_w)
            torch.cuda.synchronize()
            for k in (2, 3, 4, 5):
                assert np.array_equal(d_w[k - 2].cpu().numpy().view(np.uint64), H.reach(1, k, 9)[1]), k
            for a, b in zip(G.arrival(1, 5, 9), H.arrival(1, 5, 9)):
                assert np.array_equal(a, b)
            qs = [{"source": 1 + i % 3, "k": 4 + i % 3, "seed": i, "motif": None} for i in range(45)]
            w, _, st = batch(G, n, qs)
            assert not st.any()
            for i in range(0, 45, 4):
                assert np.array_equal(w[i], H.reach(qs[i]["source"], qs[i]["k"], i)[1]), i


def test_a_batch_of_long_queries_uses_the_whole_grid():
    # scratch for a few queries at a time (4 GB each): over the grid one after
    # another, in about the time of single queries, not on as many blocks as fit
    # (20 times that); the margin of three is for the clock
    import torch
    g = W.motif_powerlaw()
    n = g["n"]
    qs = [{"source": i, "k": 12 if i % 8 == 0 else 9, "seed": 60 + i, "motif": None} for i in range(40)]
    with capi.Graph(g) as G:
        d_w = torch.zeros((len(qs), n), dtype=torch.int64, device="cuda")
        d_1 = torch.zeros((len(qs), n), dtype=torch.int64, device="cuda")
        st = torch.cuda.current_stream().cuda_stream

        def singles():
            for i, q in enumerate(qs):
                capi.rr_reach_device(G.handle, q["source"], q["k"], q["seed"], d_1[i], None, st)

        def timed(f):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            f()
            torch.cuda.synchronize()
            a.record()
            f()
            b.record()
            torch.cuda.synchronize()
            return a.elapsed_time(b)

        one = timed(singles)
        many = timed(lambda: capi.rr_reach_batch_device(G.handle, qs, d_w, None, None, st))
        assert torch.equal(d_w, d_1) and bool(d_w.any())
        assert many < 3 * one, (many, one)


@pytest.mark.parametrize("k,scratch", [(4, 1), (7, 1), (9, 1), (9, 3_000_000), (10, 1)])
def test_calls_whose_scratch_cannot_be_had(k, scratch):
    # the engines over sieve points in their automatic shapes take what the
    # frontier engine declines (all of it, or the long queries only), with the
    # same results
    import torch
    g = W.uniform(700, 9_001, 60, 0, 12, 31 + k, ncolors=2)
    n, s = g["n"], W.first_source(g)
    motif = [int(g["color"][s])] + [i % 2 for i in range(k - 1)]
    rng = np.random.default_rng(k)
    srcs = [int(x) for x in rng.choice(n, 5, replace=False)]
    qs = [{"source": int(rng.integers(0, n)), "k": 3 + i % (k - 2), "seed": i, "motif": None} for i in range(24)]
    qs[5]["k"], qs[7]["k"] = k, 2

    def every_call(G):
        def dev(*shape, dtype=torch.int64):
            return torch.full(shape, -1, dtype=dtype, device="cuda")
        out = list(G.reach(s, k, 5)) + list(G.reach(s, k, 6, motif=motif)) + list(G.arrival(s, k, 7)) + list(G.arrival(s, k, 8, motif=motif))
        w = [dev(n), dev(k - 1, n), dev(n)]
        r, l = dev(n, dtype=torch.int32), dev(n, dtype=torch.uint8)
        capi.rr_reach_sources_device(G.handle, srcs, k, 9, w[0])
        capi.rr_reach_atmost_device(G.handle, s, k, 10, w[1])
        capi.rr_reach_bounded_device(G.handle, s, k, 11, r, l)
        capi.rr_reach_device(G.handle, s, k, 12, w[2])
        torch.cuda.synchronize()
        out += [x.cpu().numpy() for x in w] + [r.cpu().numpy(), l.cpu().numpy()]
        bw, bb, bs = batch(G, n, qs)
        reach = np.nonzero(out[2 * 2 + 2] != capi.NO_ARRIVAL)[0]
        target = int(reach[0]) if len(reach) else (s + 1) % n
        path = G.extract_path(s, k, 7, target)
        return out + [bw, bb, bs], path

    with capi.Graph(g) as G:
        want, path = every_call(G)
        assert want[1].any() and path is not None
        capi.rr_debug_frontier(G.handle, 0, 0, scratch)
        before = capi.rr_kernel_launches()
        G.reach(s, k, 5)
        assert capi.rr_kernel_launches() - before > 2  # (a frontier query: one kernel and the results')
        got, path2 = every_call(G)
        assert path2 == path
        for i, (a, b) in enumerate(zip(want, got)):
            assert np.array_equal(a, b), i
        srv = capi.rr_server_create(G.handle, 0, 2)
        try:
            ts = [capi.rr_query_submit(srv, q["source"], q["k"], q["seed"]) for q in qs]
            for i, t in enumerate(ts):
                assert np.array_equal(capi.rr_query_poll(srv, t, n)[2], want[-3][i]), i
        finally:
            capi.rr_server_destroy(srv)


@pytest.mark.parametrize("ow", [1, 4, 7])
def test_results_into_unaligned_pinned_buffers(ow):
    # witness words that do not begin on a word's boundary: the copy engine's
    import torch
    g = W.uniform(2001, 30_000, 40, 0, 6, 5)
    n, nb = g["n"], 251
    raw = torch.full((8 * n + 16,), 99, dtype=torch.uint8, pin_memory=True).numpy()
    b = torch.full((nb,), 99, dtype=torch.uint8, pin_memory=True).numpy()
    with capi.Graph(g) as G:
        b1, w1 = G.reach(1, 5, 3)
        G.reach(1, 5, 3, out=(b, raw[ow:ow + 8 * n].view(np.uint64)))
    assert np.array_equal(raw[ow:ow + 8 * n].copy().view(np.uint64), w1) and np.array_equal(b, b1) and w1.any()
    assert (raw[:ow] == 99).all() and (raw[ow + 8 * n:] == 99).all()


def hub_reads(k, p, sparse, dense, wide):
    """Edges p + 1 of the walks from vertex 0 are sparse + dense ones into a hub; each sparse one is read
    by a window of its own, and `wide` windows read all the dense ones. 300 edges of 0 lead nowhere (too
    many for one block)."""
    rows, readers = sparse + dense, sparse + wide
    chain, mid, hub = np.arange(p), p + np.arange(rows), p + rows
    out = hub + 1 + np.arange(readers)
    tail = out[-1] + 1 + np.arange(k)
    dead = tail[-1] + 1 + np.arange(300)
    t0, left = 200 + 20 * sparse, k - 3 - p  # the dense times; edges after the readers
    td = np.sort(np.random.default_rng([k, p, sparse, dense]).integers(t0, t0 + 10, dense))
    parts = [(chain[:-1], chain[1:], np.zeros(p - 1)), (np.full(rows, chain[-1]), mid, np.zeros(rows)),
             (mid, np.full(rows, hub), np.concatenate([100 + 20 * np.arange(sparse), td])),
             (np.full(readers, hub), out, np.concatenate([105 + 20 * np.arange(sparse), np.full(wide, t0 + 9)])),
             (np.zeros(300), dead, np.zeros(300))]
    if left >= 1:
        parts += [(out, np.full(readers, tail[0]), np.full(readers, t0 + 20)),
                  (tail[:left - 1], tail[1:left], t0 + 21 + np.arange(left - 1))]
    delta = np.full(int(dead[-1]) + 1, t0 + 1000)
    delta[hub] = 10
    return graph_of(*(np.concatenate([x[i] for x in parts]) for i in range(3)), delta)


@pytest.mark.parametrize("k,p,sparse,dense,wide,blocks,completed", [
    (4, 1, 10, 20, 2, (16, 47), 0), (5, 1, 10, 37, 2, (16, 47), 0),        # sums over 16 blocks
    (4, 1, 60, 60, 1, (48, 255), 0), (5, 1, 60, 60, 1, (48, 255), 0),
    (4, 1, 800, 1000, 3, (256, 4095), 0), (5, 1, 800, 1000, 3, (256, 4095), 0),  # over 256
    (12, 3, 6000, 6000, 3, (256, 4095), 0),
    (4, 1, 60, 1000, 60, (256, 4095), 1), (5, 1, 60, 1000, 60, (256, 4095), 1),  # completed: wide on average
    (4, 1, 100_000, 100_000, 3, (4096, 1 << 31), 1), (5, 1, 100_000, 100_000, 3, (4096, 1 << 31), 1),  # or long
    (12, 4, 14_000, 500, 3, (4096, 1 << 31), 1)])
def test_sums_over_blocks_and_completed_ones(k, p, sparse, dense, wide, blocks, completed):
    # (from 4,096 blocks on, sums are completed wherever a level's rows are not
    # nearly all of its list's)
    g = hub_reads(k, p, sparse, dense, wide)
    with capi.Graph(g) as G, capi.Graph(g, capi.FLAG_DENSE_STATE) as H:
        b, w = G.reach(0, k, 3)
        level, ends, rows, per, done = capi.rr_debug_levels(G.handle, k)[p]  # (one list a level)
        assert (level, ends, rows) == (p + 1, 0, sparse + dense)
        assert blocks[0] <= -(-rows // per) <= blocks[1] and done == completed
        b1, w1 = H.reach(0, k, 3)
        assert np.array_equal(w, w1) and np.array_equal(b, b1) and w.any()


@pytest.mark.parametrize("k", [2, 3, 4, 5, 6, 9, 12, 14, 16])
@pytest.mark.parametrize("dmax", [6, 25])
def test_every_size_finds_a_planted_path(k, dmax):
    # ragged sizes, a path of k vertices laid into the graph (its colours the
    # motif): a non-zero witness in every combination
    g = W.uniform(301, 3_007 if k < 14 else 1_201, 60, 0, dmax, 900 + k, ncolors=3)
    rng = np.random.default_rng([k, dmax])
    path = rng.choice(301, size=k, replace=False)
    rows = rng.choice(len(g["src"]), size=k - 1, replace=False)
    g["src"][rows], g["dst"][rows], g["t"][rows] = path[:-1], path[1:], 20 + np.arange(k - 1)
    g["delta"][path] = np.maximum(g["delta"][path], 1)
    s, end = int(path[0]), int(path[-1])
    with capi.Graph(g) as G, capi.Graph(g, capi.FLAG_DENSE_STATE) as H:
        for m in (None, g["color"][path]):
            b, w = G.reach(s, k, 77 + k, motif=m)
            b1, w1 = H.reach(s, k, 77 + k, motif=m)
            assert np.array_equal(w, w1) and np.array_equal(b, b1) and w[end]
