"""Performance cases of the restless-reachability library: what its users run.

A case is a dict of plain values: a call (``call``), a temporal graph family with
its sizes, and the query's k. ``prepare`` draws the graph and the queries from a
seed and loads the graph; ``run`` makes one call through the public binding
(paper_2010_08423_gb300.capi); ``work`` counts the bytes of the call's inputs and
outputs; ``exact`` evaluates small single queries in plain numpy.

Graph families (the library's own workload generators, drawn on the device):
  uniform   endpoints uniform, t ~ U[1, tau], delta ~ U{dmin..dmax}
  powerlaw  Chung-Lu with degree exponent gamma, t uniform or (bursts > 0) in
            Poisson(bursts) bursts of width 20
Sources: "hub" is the first vertex of a power-law graph (its largest hub); "any"
the start of a restless path of k vertices laid into the graph, so that a sparse
graph has something to find. Of many queries in one call every fourth starts at
such a path, the others at a uniformly drawn edge's tail.
"""
import math

import numpy as np
import torch

from paper_2010_08423_gb300 import capi

M64 = (1 << 64) - 1

# the temporal graphs of the library's benchmark and tests
SMALL = dict(family="uniform", n=1000, m=10_000, tau=100, dmin=1, dmax=5)
UNIFORM = dict(family="uniform", n=100_000, m=1_000_000, tau=1000, dmin=1, dmax=20)
BURSTS = dict(family="powerlaw", gamma=2.5, n=1_000_000, m=10_000_000, tau=10_000, dmin=5, dmax=50,
              bursts=50)
BURSTS_5TH = dict(BURSTS, n=200_000, m=2_000_000)
CONTACTS = dict(family="uniform", n=2000, m=30_011, tau=40, dmin=0, dmax=6)


def listed():
    return [
        # one decision query on a small network: what an interactive tool asks, all latency
        dict(SMALL, name="small_k5", call="reach", k=5, colors=0, source="any"),
        # one query on a sparse mid-size network, the kind a service answers one by one
        dict(UNIFORM, name="uniform_k8", call="reach", k=8, colors=0, source="any"),
        # the benchmark's headline: a motif query from the largest hub of a bursty power-law graph
        dict(BURSTS, name="motif_k10", call="reach", k=10, colors=8, source="hub"),
        # a long plain query from a hub, results read back to the host each time
        dict(BURSTS_5TH, name="hub_sync_k12", call="sync", k=12, colors=0, source="hub"),
        # a contact network with few people and many contacts: nearly every row takes part
        dict(CONTACTS, name="contacts_k12", call="reach", k=12, colors=0, source="any"),
        # every path length up to k from the hub of the large graph
        dict(BURSTS, name="atmost_k10", call="atmost", k=10, colors=0, source="hub"),
        # earliest arrival and shortest length over all path lengths up to k
        dict(BURSTS_5TH, name="bounded_k8", call="bounded", k=8, colors=0, source="hub"),
        # the fine-grained oracle: per-edge sums and minimum arrival times
        dict(BURSTS_5TH, name="arrival_k8", call="arrival", k=8, colors=3, source="hub"),
        # many mixed queries on one graph in one call (offline screening)
        dict(UNIFORM, name="batch_256", call="batch", k=12, kmin=4, count=256, colors=8, source="any"),
        # a burst of requests through the serving loop
        dict(UNIFORM, name="served_64", call="served", k=12, kmin=6, count=64, colors=0, source="any"),
        # one optimal path (k - 1 queries and picks in between), ragged sizes
        dict(family="uniform", n=20_011, m=200_003, tau=300, dmin=1, dmax=20, name="extract_k7",
             call="extract", k=7, colors=0, source="any"),
        # spread from an initial set of vertices with blocked ones (case study)
        dict(family="uniform", n=20_011, m=200_003, tau=300, dmin=1, dmax=20, name="sources_k6",
             call="sources", k=6, count=16, colors=0, source="any"),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: the listed calls over sizes from 1,000 to 1,000,000 vertices."""
    call = rng.choice(["reach", "reach", "reach", "sync", "atmost", "bounded", "arrival", "batch", "served",
                       "extract", "sources"])
    kind = rng.choice(["uniform", "bursts", "contacts"])
    if call in ("extract", "sources", "served"):
        kind = "uniform"
    if call == "batch" and kind == "bursts":
        kind = "uniform"
    many = call in ("batch", "served", "extract", "sources")
    if kind == "contacts":
        n = _logint(rng, 300, 3000)
        m = n * rng.randint(8, 16) + rng.randint(0, 99)
        c = dict(CONTACTS, n=n, m=m, dmax=rng.randint(3, 6))
    elif kind == "bursts":
        n = _logint(rng, 20_000, 1_000_000)
        m = min(10_000_000, n * rng.randint(6, 10) + rng.randint(0, 999))
        c = dict(BURSTS, n=n, m=m, gamma=rng.choice([2.3, 2.5]), bursts=rng.choice([0, 50, 50]))
    else:
        n = _logint(rng, 1000, 100_000 if many else 300_000)
        m = n * rng.randint(8, 10) + rng.randint(0, 999)
        c = dict(UNIFORM, n=n, m=m, tau=rng.randint(100, 1000))
    # long queries on small graphs, short ones on large: 2^k m stays below the largest listed case's
    kmax = min(12, int(math.log2(1024 * 10_000_000 / m)))
    if call == "bounded":
        kmax = min(kmax, 9)
    k = rng.randint(4, max(4, kmax))
    c.update(call=call, k=k, colors=rng.choice([0, 3, 8]) if call in ("reach", "sync", "arrival", "batch") else 0,
             source="hub" if kind == "bursts" and rng.random() < 0.7 else "any")
    if call in ("batch", "served"):
        c.update(kmin=4, count=_logint(rng, 8, 256 if call == "batch" else 64))
        c["k"] = max(k, 5)
    if call == "sources":
        c.update(count=rng.randint(2, 64))
        c["k"] = min(k, 8)
    if call == "extract":
        c["k"] = min(max(k, 5), 9)
    return c


# -- inputs ------------------------------------------------------------------

def _graph(case, seed):
    """Endpoints, times, waiting times and colours as host arrays, from the seed alone."""
    dev = torch.device("cuda")
    gen = torch.Generator(device=dev)
    gen.manual_seed(seed)
    n, m = case["n"], case["m"]

    def randint(lo, hi, size):
        return torch.randint(lo, hi, (size,), generator=gen, device=dev, dtype=torch.int64)

    if case["family"] == "uniform":
        src, dst = randint(0, n, m), randint(0, n, m)
    else:
        w = torch.arange(1, n + 1, device=dev, dtype=torch.float64) ** (-1.0 / (case["gamma"] - 1.0))
        cdf = torch.cumsum(w, 0)
        cdf /= cdf[-1].clone()

        def ends():
            return torch.searchsorted(cdf, torch.rand(m, generator=gen, device=dev, dtype=torch.float64),
                                      right=True).clamp_(max=n - 1)

        src, dst = ends(), ends()
    loop = src == dst
    dst = torch.where(loop, (dst + 1) % n, dst)  # no self-loops
    if case.get("bursts"):
        nb = max(1, int(np.random.default_rng(seed).poisson(case["bursts"])))
        centres = randint(1, case["tau"] + 1, nb)
        t = (centres[randint(0, nb, m)] + randint(0, 20, m)).clamp_(max=case["tau"])
    else:
        t = randint(1, case["tau"] + 1, m)
    delta = randint(case["dmin"], case["dmax"] + 1, n)
    color = randint(0, case["colors"], n) if case["colors"] else None

    def host(x, dtype):
        return x.to(torch.int32).cpu().numpy().astype(dtype, copy=False)

    g = {"n": n, "src": host(src, np.uint32), "dst": host(dst, np.uint32), "t": host(t, np.uint32),
         "delta": host(delta, np.uint32)}
    if color is not None:
        g["color"] = host(color, np.uint8)
    return g


def _plant(g, k, rng):
    """Overwrites k - 1 edges with a restless path of k vertices; returns the path."""
    n, m = g["n"], len(g["src"])
    path = rng.choice(n, size=k, replace=False)
    rows = rng.choice(m, size=k - 1, replace=False)
    t = int(rng.integers(1, max(2, int(g["t"].max()) - k)))
    for i, r in enumerate(rows):
        g["src"][r], g["dst"][r] = path[i], path[i + 1]
        t += int(rng.integers(0, 1 + min(3, int(g["delta"][path[i]])))) if i else 0
        g["t"][r] = t
    return path


def _query(case, g, k, rng, colored, planted):
    """A query's arguments; a motif is the source's colour plus k - 1 uniform ones, or a laid path's colours."""
    path = _plant(g, k, rng) if planted else None
    if path is not None:
        s = int(path[0])
    elif case["source"] == "hub":
        s = int(g["src"].min())
    else:
        s = int(g["src"][int(rng.integers(0, len(g["src"])))])
    motif = None
    if colored:
        rest = rng.integers(0, case["colors"], size=k - 1, dtype=np.uint8) if path is None else g["color"][path[1:]]
        motif = np.concatenate([np.array([g["color"][s]], dtype=np.uint8), rest])
    return {"source": s, "k": k, "seed": int(rng.integers(1, 1 << 63)), "motif": motif}, path


def _inputs(case, seed):
    """The graph, the call's queries and a generator for what else the call takes."""
    rng = np.random.default_rng([seed, case["n"], case["m"], case["k"]])
    g = _graph(case, seed & 0x7FFFFFFF)
    if case["call"] in ("batch", "served"):
        made = [_query(case, g, int(rng.integers(case["kmin"], case["k"] + 1)), rng,
                       bool(case["colors"]) and i % 2 == 1, i % 4 == 3) for i in range(case["count"])]
    else:
        made = [_query(case, g, case["k"], rng, bool(case["colors"]), case["source"] == "any")]
    return g, [q for q, _ in made], made[0][1], rng


class _Owner:
    """The loaded graph (and server) of a state, freed with it."""

    def __init__(self, g):
        self.graph = capi.Graph(g)
        self.server = None

    def __del__(self):
        if self.server is not None:
            capi.rr_server_destroy(self.server)
        self.graph.close()


def prepare(case, seed):
    g, queries, path, rng = _inputs(case, seed)
    n, m, k, call = case["n"], case["m"], case["k"], case["call"]
    st = {"case": case, "g": g, "queries": queries, "q": queries[0]}
    if call == "extract":
        st["target"] = int(path[-1])
    if call == "sources":
        picked = rng.choice(n, size=case["count"] - 1 + max(1, n // 100), replace=False).astype(np.uint32)
        st["sources"] = np.concatenate([np.array([path[0]], dtype=np.uint32), picked[:case["count"] - 1]])
        sep = np.zeros(n, dtype=np.uint8)
        sep[picked[case["count"] - 1:]] = 1
        sep[path] = 0
        st["separators"] = torch.from_numpy(sep).cuda()
    own = st["own"] = _Owner(g)
    st["h"] = own.graph.handle
    dev, nb = "cuda", (n + 7) // 8
    if call in ("reach", "sources", "arrival"):
        st["w"] = torch.empty(n, dtype=torch.int64, device=dev)
        st["b"] = torch.empty(nb, dtype=torch.uint8, device=dev)
    if call == "sync":
        st["hw"] = torch.empty(n, dtype=torch.int64, pin_memory=True)
        st["hb"] = torch.empty(nb, dtype=torch.uint8, pin_memory=True)
    if call == "arrival":
        st["e"] = torch.empty(m, dtype=torch.int64, device=dev)
        st["r"] = torch.empty(n, dtype=torch.int32, device=dev)
    if call == "atmost":
        st["w"] = torch.empty((k - 1, n), dtype=torch.int64, device=dev)
        st["b"] = torch.empty(nb, dtype=torch.uint8, device=dev)
    if call == "bounded":
        st["r"] = torch.empty(n, dtype=torch.int32, device=dev)
        st["l"] = torch.empty(n, dtype=torch.uint8, device=dev)
        st["b"] = torch.empty(nb, dtype=torch.uint8, device=dev)
    if call == "batch":
        st["w"] = torch.empty((case["count"], n), dtype=torch.int64, device=dev)
        st["b"] = torch.empty((case["count"], nb), dtype=torch.uint8, device=dev)
        st["s"] = torch.empty(case["count"], dtype=torch.int32, device=dev)
    if call == "served":
        own.server = capi.rr_server_create(st["h"], 0, 4)
    return st


def run(st):
    call, h = st["case"]["call"], st["h"]
    n, k = st["case"]["n"], st["case"]["k"]
    stream = torch.cuda.current_stream().cuda_stream
    q = st["q"]
    if call == "extract":
        path = capi.rr_extract_path(h, q["source"], k, q["seed"], st["target"])
        return [np.asarray(x, dtype=np.int64) for x in path]
    if call == "batch":
        capi.rr_reach_batch_device(h, st["queries"], st["w"], st["b"], st["s"], stream)
        return [st["w"], st["b"], st["s"]]
    if call == "served":
        srv = st["own"].server
        tickets = [capi.rr_query_submit(srv, q["source"], q["k"], q["seed"]) for q in st["queries"]]
        done = [capi.rr_query_poll(srv, t, n) for t in tickets]
        return [np.array([d[0] for d in done], dtype=np.int64), np.stack([d[1] for d in done]),
                np.stack([d[2] for d in done]).view(np.int64)]
    if call == "reach":
        capi.rr_reach_device(h, q["source"], k, q["seed"], st["w"], st["b"], stream, q["motif"])
        return [st["w"], st["b"]]
    if call == "sync":
        capi.rr_reach_sync(h, n, q["source"], k, q["seed"], q["motif"],
                           out=(st["hb"].numpy(), st["hw"].numpy().view(np.uint64)))
        return [st["hw"], st["hb"]]
    if call == "arrival":
        capi.rr_reach_arrival_device(h, q["source"], k, q["seed"], st["w"], st["r"], st["e"], st["b"], stream,
                                     q["motif"])
        return [st["w"], st["e"], st["r"], st["b"]]
    if call == "atmost":
        capi.rr_reach_atmost_device(h, q["source"], k, q["seed"], st["w"], st["b"], stream)
        return [st["w"], st["b"]]
    if call == "bounded":
        capi.rr_reach_bounded_device(h, q["source"], k, q["seed"], st["r"], st["l"], st["b"], stream)
        return [st["r"], st["l"], st["b"]]
    if call == "sources":
        capi.rr_reach_sources_device(h, st["sources"], k, q["seed"], st["w"], st["b"], st["separators"], stream)
        return [st["w"], st["b"]]
    raise ValueError(call)


def work(case):
    """The graph's arrays read once and the outputs written once. The arithmetic is in GF(2^64), on
    integer instructions: no floating-point operations."""
    n, m, k, call = case["n"], case["m"], case["k"], case["call"]
    nb = (n + 7) // 8
    graph = 12 * m + 4 * n + (n if case["colors"] else 0)
    out = {"reach": 8 * n + nb, "sync": 8 * n + nb, "sources": 9 * n + nb, "arrival": 8 * m + 12 * n + nb,
           "atmost": 8 * n * (k - 1) + nb, "bounded": 5 * n + nb, "extract": 12 * k,
           "batch": case.get("count", 0) * (8 * n + nb), "served": case.get("count", 0) * (8 * n + nb)}[call]
    return {"bytes": graph + out, "flops": 0}


# -- the definition in plain numpy ---------------------------------------------

def _mul(a, b):
    """Products in GF(2)[x]/(x^64 + x^4 + x^3 + x + 1) of uint64 arrays (broadcast)."""
    a, b = np.broadcast_arrays(a, b)
    a, r = a.copy(), np.zeros(a.shape, dtype=np.uint64)
    one = np.uint64(1)
    for i in range(64):
        r ^= a * ((b >> np.uint64(i)) & one)
        a = (a << one) ^ ((a >> np.uint64(63)) * np.uint64(0x1B))
    return r


def _mix(z):
    z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
    z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
    return z ^ (z >> np.uint64(31))


def _draws(seed, tag, index):
    key = _mix(np.array((seed ^ tag) & M64, dtype=np.uint64))
    return _mix(key + (index.astype(np.uint64) + np.uint64(1)) * np.uint64(0x9E3779B97F4A7C15))


def exact(case, seed):
    """Small single queries by the definition: every sieve point, layer by layer."""
    k, n = case["k"], case["n"]
    if case["call"] not in ("reach", "sync") or (k * case["m"]) << k > 8_000_000:
        return None
    g, (q,), _, _ = _inputs(case, seed)
    with np.errstate(over="ignore"):
        # rows by head, then time; row e's window lies in its tail's rows
        order = np.lexsort((g["t"], g["dst"]))
        src, dst, t = (g[x][order].astype(np.int64) for x in ("src", "dst", "t"))
        pos = dst * (1 << 32) + t
        lo = np.searchsorted(pos, src * (1 << 32) + np.maximum(t - g["delta"][src], 0), "left")
        hi = np.maximum(lo, np.searchsorted(pos, src * (1 << 32) + t, "right"))
        if q["motif"] is None:
            z = _draws(q["seed"], 2, np.arange(n)[:, None] * 32 + np.arange(k))
        else:
            z = np.zeros((n, k), dtype=np.uint64)
            for d, c in enumerate(np.sort(q["motif"])):
                own = np.nonzero(g["color"] == c)[0]
                z[own] ^= _mul(_draws(q["seed"], 3, own * 32 + d)[:, None], _draws(q["seed"], 4, d * 32 + np.arange(k)))
        bits = (np.arange(1 << k)[:, None] >> np.arange(k)) & 1
        x = np.zeros((1 << k, n), dtype=np.uint64)
        for j in range(k):
            x ^= np.where(bits[:, j:j + 1] != 0, z[:, j], np.uint64(0))
        p = None
        for layer in range(1, k):
            y = _draws(q["seed"], 1, order * 32 + (layer - 1))
            if p is None:
                w = np.where(src == q["source"], x[:, q["source"]][:, None], np.uint64(0))
            else:
                acc = np.zeros((p.shape[0], p.shape[1] + 1), dtype=np.uint64)
                np.bitwise_xor.accumulate(p, axis=1, out=acc[:, 1:])
                w = acc[:, hi] ^ acc[:, lo]
            p = _mul(_mul(x[:, dst], y), w)
        sums = np.bitwise_xor.reduce(p, axis=0)
        out = np.zeros(n, dtype=np.uint64)
        np.bitwise_xor.at(out, dst, sums)
    return [out.view(np.int64), np.packbits(out != 0, bitorder="little")]
