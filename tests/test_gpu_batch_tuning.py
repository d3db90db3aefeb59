"""A batch shape chosen by rr_set_batch_tuning keeps whole batches on the
persistent sieve-point kernel, before and after a tuning call."""
import numpy as np
import pytest

from paper_2010_08423_gb300 import capi
from paper_2010_08423_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def test_a_chosen_shape_holds_after_tuning():
    import torch
    torch.cuda.set_device(0)
    capi.load()
    g = W.uniform(300, 3_001, 40, 0, 8, 17)
    n = g["n"]
    qs = [{"source": 7 * i, "k": 4 + i % 4, "seed": i, "motif": None} for i in range(6)]
    with capi.Graph(g) as G:
        d_w = torch.zeros((6, n), dtype=torch.int64, device="cuda")

        def run():
            before = capi.rr_kernel_launches()
            capi.rr_reach_batch_device(G.handle, qs, d_w)
            torch.cuda.synchronize()
            return capi.rr_kernel_launches() - before, d_w.cpu().numpy()

        free, want = run()
        assert free == 1  # the frontier engine's one launch
        capi.rr_autotune_batch(G.handle, qs)
        assert run()[0] == 1  # nothing chosen: still its choice
        capi.rr_set_batch_tuning(G.handle, 2, 1, 256)
        assert run()[0] > 1
        capi.rr_autotune_batch(G.handle, qs)
        count, got = run()
        assert count > 1 and np.array_equal(got, want) and want.any()
        capi.rr_set_batch_tuning(G.handle)
        assert run()[0] == 1
