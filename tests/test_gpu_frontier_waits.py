"""Failure path of the bounded waits inside a whole query's kernel, tested
without a GPU fault.

The blocks of such a kernel meet at barriers whose waits end after a limit.
rr_debug_frontier lets the last block leave before a meeting, so that the others
wait in vain for a few milliseconds: the query must then be reported -- by the
call itself, by its status, by the next call or by its ticket, and once --, and
the context must stay usable.
"""
import numpy as np
import pytest

import oracle
from paper_2010_08423_gb300 import capi
from paper_2010_08423_gb300 import workloads as W

pytestmark = pytest.mark.gpu
LIMIT = 3_000_000  # ns


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    capi.load()
    oracle.build()
    torch.cuda.set_device(0)


@pytest.fixture()
def graph():
    g = W.uniform(300, 5_001, 40, 0, 8, 17)
    with capi.Graph(g) as G:
        yield g, G


def usable(g, G, k=5):
    assert np.array_equal(G.reach(3, k, 11)[1], oracle.sieve(g, 3, k, 11))


def test_a_synchronous_query_reports_itself(graph):
    g, G = graph
    usable(g, G)
    for _ in range(2):
        capi.rr_debug_frontier(G.handle, LIMIT, 1)
        with pytest.raises(capi.RRError) as ei:
            G.reach(3, 7, 1)
        assert ei.value.status == capi.RR_ETIMEDOUT
        capi.rr_debug_frontier(G.handle)
        usable(g, G)


def test_an_enqueued_query_is_reported_once(graph):
    import torch
    g, G = graph
    d_w = torch.zeros(g["n"], dtype=torch.int64, device="cuda")
    calls = [lambda: capi.rr_reach_device(G.handle, 3, 7, 1, d_w),
             lambda: capi.rr_reach_batch_device(G.handle, [{"source": 3, "k": 7, "seed": 1, "motif": None}] * 2,
                                                torch.zeros((2, g["n"]), dtype=torch.int64, device="cuda"))]
    for call in calls:
        capi.rr_debug_frontier(G.handle, LIMIT, 1)
        call()
        torch.cuda.synchronize()
        capi.rr_debug_frontier(G.handle)
        # a batch with statuses is not refused for it, and leaves it to the next call
        b_w = torch.zeros((1, g["n"]), dtype=torch.int64, device="cuda")
        b_s = torch.full((1,), -1, dtype=torch.int32, device="cuda")
        capi.rr_reach_batch_device(G.handle, [{"source": 3, "k": 5, "seed": 11, "motif": None}], b_w, None, b_s)
        torch.cuda.synchronize()
        assert int(b_s) == 0 and np.array_equal(b_w[0].cpu().numpy().view(np.uint64), oracle.sieve(g, 3, 5, 11))
        with pytest.raises(capi.RRError) as ei:
            capi.rr_reach_device(G.handle, 3, 5, 11, d_w)
        assert ei.value.status == capi.RR_ETIMEDOUT
        usable(g, G)


@pytest.mark.parametrize("absent", [1, 2])
@pytest.mark.parametrize("mixed", [False, True])
def test_a_batch_marks_its_unfinished_queries(graph, absent, mixed):
    # queries from vertices without edges end in one block (done before the
    # second meeting); k = 17 goes to the sieve-point engine; nothing is left for
    # the next call
    import torch
    g, _ = graph
    alone = np.arange(300, 320)
    g = dict(g, n=320, delta=np.concatenate([g["delta"], np.ones(20, np.uint32)]))
    with capi.Graph(g) as G:
        n = g["n"]
        qs = [{"source": int(alone[i % 20]) if i % 3 == 0 else (5 * i) % 300, "k": 7 + i % 3, "seed": i, "motif": None}
              for i in range(30)]
        if mixed:
            qs[4] = {"source": 3, "k": 17, "seed": 8, "motif": None}
        d_w = torch.full((30, n), -1, dtype=torch.int64, device="cuda")
        d_s = torch.full((30,), -1, dtype=torch.int32, device="cuda")
        capi.rr_debug_frontier(G.handle, LIMIT, absent)
        capi.rr_reach_batch_device(G.handle, qs, d_w, None, d_s)
        torch.cuda.synchronize()
        st = d_s.cpu().numpy()
        for i, q in enumerate(qs):
            done = q["k"] == 17 or (absent == 2 and i % 3 == 0)
            assert st[i] == (0 if done else capi.RR_ETIMEDOUT), i
        capi.rr_debug_frontier(G.handle)
        w17 = d_w[4].cpu().numpy().view(np.uint64)
        usable(g, G)  # the next call is not refused
        if mixed:
            assert np.array_equal(w17, G.reach(3, 17, 8)[1])
        capi.rr_reach_batch_device(G.handle, qs, d_w, None, d_s)
        torch.cuda.synchronize()
        assert not d_s.cpu().numpy().any()
        for i in (0, 1, 2, 4, 29):
            assert np.array_equal(d_w[i].cpu().numpy().view(np.uint64), G.reach(qs[i]["source"], qs[i]["k"], qs[i]["seed"])[1])


@pytest.mark.parametrize("batches", [False, True])
def test_served_tickets_fail_and_the_server_goes_on(graph, batches):
    g, G = graph
    srv = capi.rr_server_create(G.handle, 0, 2)
    try:
        if batches:
            capi.rr_server_set_batching(srv, 8, 16)
        capi.rr_debug_frontier(G.handle, LIMIT, 1)
        tickets = [capi.rr_query_submit(srv, 3, 7, i) for i in range(24)]
        for t in tickets:
            with pytest.raises(capi.RRError) as ei:
                capi.rr_query_poll(srv, t, g["n"])
            assert ei.value.status in (capi.RR_ETIMEDOUT, capi.RR_ECUDA)
        capi.rr_debug_frontier(G.handle)
        tickets = [capi.rr_query_submit(srv, 3, 5, 11) for _ in range(24)]
        ref = oracle.sieve(g, 3, 5, 11)
        for t in tickets:
            st, _, w = capi.rr_query_poll(srv, t, g["n"])
            assert st == capi.RR_OK and np.array_equal(w, ref)
        usable(g, G)
        if batches:
            assert capi.rr_server_stats(srv)[1] > 0
    finally:
        capi.rr_server_destroy(srv)


def test_argument_errors(graph):
    _, G = graph
    for args in ((20_000_000_000, 0), (0, 3)):
        with pytest.raises(capi.RRError) as ei:
            capi.rr_debug_frontier(G.handle, *args)
        assert ei.value.status == capi.RR_EINVAL


def test_queries_on_lanes_are_reported_once(graph):
    # at-most-k whose own scratch cannot be had runs its queries on lanes, which
    # take the frontier engine where a single query's scratch can be had
    import torch
    g, G = graph
    k, n = 7, g["n"]
    d_w = torch.zeros((k - 1, n), dtype=torch.int64, device="cuda")

    def atmost():
        before = capi.rr_kernel_launches()
        capi.rr_reach_atmost_device(G.handle, 3, k, 11, d_w)
        torch.cuda.synchronize()
        return capi.rr_kernel_launches() - before

    def launches(scratch):
        capi.rr_debug_frontier(G.handle, 0, 0, scratch)
        return atmost()

    want = launches(0) and d_w.cpu().numpy()
    lo, hi = 1, 1 << 34  # the least scratch for which at-most-k is one launch
    while lo < hi:
        mid = (lo + hi) // 2
        lo, hi = (lo, mid) if launches(mid) == 1 else (mid + 1, hi)
    assert launches(lo) == 1 and launches(lo - 1) == k - 1  # one frontier query a lane
    assert np.array_equal(d_w.cpu().numpy(), want)
    d_r = torch.zeros(n, dtype=torch.int32, device="cuda")
    for call in (atmost, lambda: capi.rr_reach_bounded_device(G.handle, 3, k, 11, d_r)):
        for again in (atmost, lambda: usable(g, G)):
            capi.rr_debug_frontier(G.handle, LIMIT, 1, lo - 1)
            call()
            torch.cuda.synchronize()
            capi.rr_debug_frontier(G.handle, 0, 0, lo - 1)
            with pytest.raises(capi.RRError) as ei:
                again()
            assert ei.value.status == capi.RR_ETIMEDOUT
            usable(g, G)
            assert atmost() == k - 1 and np.array_equal(d_w.cpu().numpy(), want)
