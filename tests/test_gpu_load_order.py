"""A walk on a non-blocking stream directly after a load: nothing of the load
may still be queued then (a cursor cleared under the walk hands queries out
twice, counters cleared or filled late do not add up)."""

import pytest
import torch

import fw_inputs as fi
from gpu_common import cached_graph, device_graph, recount

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("borrow", [False, True])
@pytest.mark.parametrize("mode", ["exact", "fast"])
def test_walk_on_a_side_stream_right_after_the_load(mode, borrow):
    g = cached_graph("rmat", 12, 2).to("cuda")
    side = torch.cuda.Stream()
    starts = fi.random_starts(g.n, 5000, 3, "cuda")
    ref = device_graph(g)
    want = ref.walk("weighted", starts, 6, 11, mode=mode)
    torch.cuda.synchronize()
    for _ in range(50):
        dg = device_graph(g, borrow=borrow)
        paths, plen = dg.walk("weighted", starts, 6, 11, mode=mode, stream=side)
        st = dg.stats()
        assert torch.equal(paths, want[0]) and torch.equal(plen, want[1])
        assert st["walks"] == starts.numel()
        assert (st["steps"], st["rows_scanned"]) == recount(g, paths, plen)
        assert st["warp_steps"] + st["block_steps"] == st["steps"]
        dg.free()
