"""A served request is complete only when every lane's padding is written: walks
that end at once in wide path rows, in arena space that longer walks have
filled before, must come back padded to the end."""

import pytest
import torch

import fw_inputs as fi
from gpu_common import cached_graph, check_valid, device_graph

pytestmark = [pytest.mark.gpu, pytest.mark.timeout(180)]


@pytest.mark.parametrize("width", [31, 100, 3000])
def test_padding_is_written_before_completion(width):
    from paper_2404_08364_gb300 import Server
    g = cached_graph("rmat", 12, 2)
    srv = Server(device_graph(g), mode="fast", mem_budget=8 << 20)
    n_q = 40
    starts = fi.random_starts(g.n, n_q, 7)
    none = torch.arange(n_q, dtype=torch.int32) % 3  # 0, 1 or 2 moves
    for i in range(30):
        full = srv.submit("weighted", starts, width, 100 + i)
        check_valid(g, *(t.cuda() for t in srv.result(full)[:2]), "weighted")
        ended = [srv.submit("weighted", starts, width, 200 + i, lengths=none) for _ in range(4)]
        for t in ended:
            paths, plen, _ = srv.result(t)
            assert bool((plen <= none + 1).all())
            check_valid(g, paths.cuda(), plen.cuda(), "weighted")  # padding is -1
    srv.close()
