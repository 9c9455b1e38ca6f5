"""Batched walks while another walk of the same graph still runs: both add to
the graph's counters, and neither's counts may be lost."""

import pytest
import torch

import fw_inputs as fi
from gpu_common import cached_graph, device_graph, recount

pytestmark = pytest.mark.gpu


def test_batched_beside_a_running_walk():
    g = cached_graph("rmat", 14, 2)
    dg = device_graph(g)
    side = torch.cuda.Stream()
    big = fi.random_starts(g.n, 60000, 1, "cuda")
    small = fi.random_starts(g.n, 500, 2)
    torch.cuda.synchronize()
    for _ in range(10):
        dg.stats_reset()
        torch.cuda.synchronize()
        a = dg.walk("weighted", big, 20, 5, mode="fast", stream=side)
        p, l, _ = dg.walk_batched("weighted", small, 4, 6, mode="fast", budget_bytes=1 << 16)
        torch.cuda.synchronize()
        st = dg.stats()
        e = [recount(g, x.cuda(), y.cuda()) for x, y in (a, (p, l))]
        assert st["walks"] == 60500
        assert (st["steps"], st["rows_scanned"]) == (e[0][0] + e[1][0], e[0][1] + e[1][1])
