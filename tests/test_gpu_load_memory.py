"""A graph that fits the device only without the frontier engine's arrays is
loaded without them, and its queries run over sieve points."""
import numpy as np
import pytest

from paper_2010_08423_gb300 import capi
from paper_2010_08423_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def test_the_smallest_memory_a_graph_loads_in():
    import torch
    torch.cuda.set_device(0)
    capi.load()
    g = W.uniform(150_000, 3_000_000, 1000, 5, 60, 77)
    s = W.first_source(g)
    with capi.Graph(g) as G:
        full = G.info()["device_bytes"]
        want = G.reach(s, 6, 1)
        assert want[1].any()

    def load(mib):
        """The graph with `mib` MiB of device memory free, or None."""
        torch.cuda.empty_cache()
        hog = torch.empty(torch.cuda.mem_get_info()[0] - (mib << 20), dtype=torch.uint8, device="cuda")
        try:
            return capi.Graph(g)
        except capi.RRError as e:
            assert e.status == capi.RR_ENOMEM
            return None
        finally:
            del hog
            torch.cuda.empty_cache()

    lo, hi = 16, 4096  # MiB
    while lo < hi:
        mid = (lo + hi) // 2
        G = load(mid)
        if G is None:
            lo = mid + 1
        else:
            G.close()
            hi = mid
    with load(lo) as G:
        assert G.info()["device_bytes"] < full - 20 * len(g["src"])
        bm, w = G.reach(s, 6, 1)
        assert np.array_equal(w, want[1]) and np.array_equal(bm, want[0])
    with load(lo + 1024) as G:
        assert G.info()["device_bytes"] == full
        assert np.array_equal(G.reach(s, 6, 1)[1], want[1])
