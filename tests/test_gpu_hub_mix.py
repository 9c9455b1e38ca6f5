"""Rows of many different segment counts in the CTA sampler at once: a hub
task's entry is taken again as soon as its last segment is merged, by a task of
another count, while warps still hold results of the one before.  The walks
have to be those of a launch that shares no row."""

import pytest
import torch

from gpu_common import built, need_gpu

pytestmark = pytest.mark.gpu

HUB_ROWS = (16400, 20000, 33000, 40000, 49200, 66000, 100000, 139000)


def hub_graph():
    """Eight hubs, whose rows hold other leaves each; every leaf's row holds
    all hubs: a walk alternates between hubs and leaves."""
    leaves, hubs = 140000, len(HUB_ROWS)
    n = hubs + leaves
    rows = [hubs + (torch.arange(d) * (leaves // d) if 2 * d <= leaves else torch.arange(d)) for d in HUB_ROWS]
    col = torch.cat(rows + [torch.arange(hubs).repeat(leaves)]).to(torch.int32)
    deg = torch.tensor([len(r) for r in rows] + [hubs] * leaves)
    row_ptr = torch.zeros(n + 1, dtype=torch.int64)
    row_ptr[1:] = deg.cumsum(0)
    w = 1 + torch.arange(col.numel(), dtype=torch.int64) * 2654435761 % 4
    return n, row_ptr, col, w.to(torch.float32), w.to(torch.int32)


@pytest.mark.parametrize("algo", ["weighted", "node2vec"])
@pytest.mark.parametrize("mode", ["fast", "exact"])
def test_shared_rows_of_many_sizes(algo, mode):
    need_gpu()
    built()
    from paper_2404_08364_gb300 import DeviceGraph
    n, row_ptr, col, w_f32, w_u32 = hub_graph()
    dg = DeviceGraph.from_tensors(row_ptr, col, w_f32, w_u32)
    n_q, L = 20000, 9
    starts = (torch.arange(n_q, dtype=torch.int32) % len(HUB_ROWS)).cuda()
    kw = dict(mode=mode, p=2.0, q=0.5)
    dg.set_tuning(d_warp=1 << 30)
    want = dg.walk(algo, starts, L, 5, **kw)
    torch.cuda.synchronize()
    for tuning in (dict(d_warp=1024), dict(block_threads=512, slots=64, d_warp=1024)):
        dg.set_tuning(**tuning)
        dg.stats_reset()
        got = dg.walk(algo, starts, L, 5, **kw)
        st = dg.stats()
        assert all(torch.equal(a, b) for a, b in zip(got, want))
        assert st["block_steps"] == n_q * 5 and st["steps"] == n_q * L
