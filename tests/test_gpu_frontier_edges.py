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
