"""GPU parity of the frontier engine at the edges of its two paths.

A query whose walks are few runs in one block's shared memory (at most 256
rows a layer); any other goes through the bitmap passes, whose rows are kept as
prefix sums in blocks with sums over 16 and 256 blocks. Both must equal the
per-point engine (the dense-layout load flag) and the oracle bit for bit.
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


def _fan(width, tails=3, n_extra=5):
    """0 -> width mid vertices -> tails sinks -> one vertex, restless throughout."""
    mid = np.arange(1, width + 1)
    sink = width + 1 + np.arange(tails)
    end = width + 1 + tails
    src = np.concatenate([np.zeros(width, int), np.repeat(mid, tails), sink])
    dst = np.concatenate([mid, np.tile(sink, width), np.full(tails, end)])
    t = np.concatenate([np.full(width, 3), np.full(width * tails, 4), np.full(tails, 6)])
    n = end + 1 + n_extra
    return {"n": n, "src": src.astype(np.uint32), "dst": dst.astype(np.uint32), "t": t.astype(np.uint32),
            "delta": np.full(n, 2, np.uint32), "color": (np.arange(n) % 2).astype(np.uint8)}


@pytest.mark.parametrize("width,tails", [(1, 1), (31, 4), (42, 3), (43, 3), (127, 1), (128, 1), (129, 1), (64, 2), (65, 2),
                                         (85, 3), (86, 3), (255, 1), (256, 1), (257, 1), (128, 2), (129, 2)])
def test_rows_around_the_block_limit(width, tails):
    # 127 .. 257 rows at layer 1, 126 .. 258 at layer 2: word and limit edges
    g = _fan(width, tails)
    with capi.Graph(g) as G:
        for k in (2, 3, 4):
            _, w = G.reach(0, k, 11 * width + k)
            assert np.array_equal(w, oracle.sieve(g, 0, k, 11 * width + k)), k
            assert w.any()
        S, E, R, _ = G.arrival(0, 4, 5)
        ref, refE = oracle.sieve(g, 0, 4, 5, edges=True)
        assert np.array_equal(S, ref) and np.array_equal(E, refE)
        assert np.array_equal(R, oracle.arrival_times(g, refE))


@pytest.mark.parametrize("k", [2, 3, 4, 5, 6, 9, 12, 14, 16])
@pytest.mark.parametrize("dmax", [6, 25])
def test_every_size_equals_the_per_point_engine(k, dmax):
    # ragged sizes; with the long waits hundreds to thousands of rows a layer
    # (the bitmap passes), with the short ones few
    g = W.uniform(301, 3_007 if k < 14 else 1_201, 60, 0, dmax, 900 + k, ncolors=3)
    s = W.first_source(g)
    motif = W.motif_for(g, s, k, 5, ncolors=3)
    with capi.Graph(g) as G, capi.Graph(g, capi.FLAG_DENSE_STATE) as H:
        for m in (None, motif):
            _, w = G.reach(s, k, 77 + k, motif=m)
            _, ref = H.reach(s, k, 77 + k, motif=m)
            assert np.array_equal(w, ref)
            assert w.any() or m is not None or dmax == 6 or k > 12


@pytest.mark.parametrize("k", [13, 14, 15, 16])
def test_long_paths_in_a_small_crowd(k):
    # 24 vertices, long waits: thousands of values a row
    g = W.uniform(24, 500 + k, 80, 30, 80, 40 + k)
    with capi.Graph(g) as G, capi.Graph(g, capi.FLAG_DENSE_STATE) as H:
        _, w = G.reach(3, k, k)
        _, ref = H.reach(3, k, k)
        assert np.array_equal(w, ref) and w.any()


@pytest.mark.parametrize("rows", [300, 5_000, 40_000])
def test_windows_over_many_blocks(rows):
    # `rows` edges from distinct tails into vertex 1, read by wide and narrow
    # windows: sums over blocks, 16 and 256 blocks and their ends
    rng = np.random.default_rng(rows)
    mid = 2 + np.arange(rows)
    out = 2 + rows + np.arange(60)
    src = np.concatenate([np.zeros(rows, int), mid, np.ones(60, int), out])
    dst = np.concatenate([mid, np.ones(rows, int), out, np.full(60, out[-1] + 1)])
    t = np.concatenate([np.zeros(rows, int), np.sort(rng.integers(1, 1000, rows)), rng.integers(1, 1400, 60),
                        np.full(60, 1500)])
    n = int(out[-1]) + 2
    delta = np.full(n, 2000)
    delta[1] = 350
    g = {"n": n, "src": src.astype(np.uint32), "dst": dst.astype(np.uint32), "t": t.astype(np.uint32),
         "delta": delta.astype(np.uint32)}
    with capi.Graph(g) as G:
        for k in (3, 4, 5):
            _, w = G.reach(0, k, 31 + k)
            assert np.array_equal(w, oracle.sieve(g, 0, k, 31 + k)), k
            assert w.any()


@pytest.mark.parametrize("nq", [1, 5, 60])
def test_batches_whose_queries_fill_the_rows(nq):
    # no query fits one block's memory: few go one after another over the whole
    # grid, many one per block; one with k = 17 goes to the per-point engine
    import torch
    g = W.uniform(300, 5_001, 40, 0, 8, 17, ncolors=2)
    n = g["n"]
    qs = W.query_set(g, nq, 4, 9, 99, ncolors=2)
    if nq == 5:
        qs[2] = {"source": 3, "k": 17, "seed": 8, "motif": None}
    with capi.Graph(g) as G:
        d_w = torch.full((nq, n), -1, dtype=torch.int64, device="cuda")
        d_b = torch.full((nq, (n + 7) // 8), 255, dtype=torch.uint8, device="cuda")
        d_s = torch.full((nq,), -1, dtype=torch.int32, device="cuda")
        for _ in range(2):
            capi.rr_reach_batch_device(G.handle, qs, d_w, d_b, d_s)
        torch.cuda.synchronize()
        assert not d_s.cpu().numpy().any()
        w = d_w.cpu().numpy().view(np.uint64)
        bm = d_b.cpu().numpy()
        for i, q in enumerate(qs):
            b1, w1 = G.reach(q["source"], q["k"], q["seed"], motif=q["motif"])
            assert np.array_equal(w[i], w1) and np.array_equal(bm[i], b1), i
            if q["k"] <= 6:
                assert np.array_equal(w1, oracle.sieve(g, q["source"], q["k"], q["seed"], motif=q["motif"])), i


def test_long_queries_one_after_another():
    # 37 queries of 14 to 16 vertices that no block's memory holds: a launch whose
    # blocks meet some 2,000 times, 300,000 arrivals
    import torch
    g = W.uniform(300, 5_001, 40, 0, 8, 17, ncolors=2)
    n = g["n"]
    nq = 37
    qs = [{"source": (7 * i) % n, "k": 14 + i % 3, "seed": 100 + i, "motif": None} for i in range(nq)]
    with capi.Graph(g) as G:
        d_w = torch.full((nq, n), -1, dtype=torch.int64, device="cuda")
        d_b = torch.full((nq, (n + 7) // 8), 255, dtype=torch.uint8, device="cuda")
        d_s = torch.full((nq,), -1, dtype=torch.int32, device="cuda")
        capi.rr_reach_batch_device(G.handle, qs, d_w, d_b, d_s)
        torch.cuda.synchronize()
        assert not d_s.cpu().numpy().any()
        w = d_w.cpu().numpy().view(np.uint64)
        for i in range(0, nq, 6):
            _, w1 = G.reach(qs[i]["source"], qs[i]["k"], qs[i]["seed"])
            assert np.array_equal(w[i], w1), i
        assert w.any()


@pytest.mark.parametrize("n,ow,ob", [(33, 0, 0), (37, 1, 1), (2000, 0, 3), (2001, 1, 16), (4097, 2, 0)])
def test_results_into_pinned_buffers(n, ow, ob):
    # one kernel writes both; every alignment, words and bytes left over, and
    # nothing beyond them
    import torch
    g = W.uniform(n, 15 * n, 40, 0, 6, 5)
    nb = (n + 7) // 8
    w = torch.full((n + ow + 2,), -7, dtype=torch.int64, pin_memory=True).numpy().view(np.uint64)
    b = torch.full((nb + ob + 2,), 99, dtype=torch.uint8, pin_memory=True).numpy()
    with capi.Graph(g) as G:
        b1, w1 = G.reach(1, 5, 3)
        G.reach(1, 5, 3, out=(b[ob:ob + nb], w[ow:ow + n]))
    assert np.array_equal(w[ow:ow + n], w1) and np.array_equal(b[ob:ob + nb], b1)
    assert w1.any()
    assert (w[:ow].view(np.int64) == -7).all() and (w[ow + n:].view(np.int64) == -7).all()
    assert (b[:ob] == 99).all() and (b[ob + nb:] == 99).all()
