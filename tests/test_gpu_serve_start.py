"""A request submitted the moment its server exists: nothing of the server's
set-up may still be queued then (a published count cleared late loses the
request)."""

import pytest
import torch

import fw_inputs as fi
from gpu_common import cached_graph, device_graph

pytestmark = [pytest.mark.gpu, pytest.mark.timeout(180)]


@pytest.mark.parametrize("mode", ["exact", "fast"])
def test_first_request_right_after_creation(mode):
    from paper_2404_08364_gb300 import Server
    g = cached_graph("rmat", 12, 2)
    dg = device_graph(g)
    starts = fi.random_starts(g.n, 300, 5)
    want = [t.cpu() for t in dg.walk("weighted", starts.cuda(), 10, 9, mode=mode)]
    for _ in range(40):
        srv = Server(dg, mode=mode, mem_budget=4 << 20, max_requests=4)
        paths, plen, _ = srv.result(srv.submit("weighted", starts, 10, 9), timeout_s=20.0)
        st = srv.stats()
        srv.close()
        assert torch.equal(paths, want[0]) and torch.equal(plen, want[1])
        assert st["completed"] == 1
