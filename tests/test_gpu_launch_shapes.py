"""Launches around the sizes where the CTA shape changes (24 and 32 walks per
SM, on a graph with rows to share): a query's path depends on its id alone, so
every launch's paths are the first rows of a larger one's."""

import pytest
import torch

from gpu_common import built, need_gpu
from test_gpu_hub_mix import HUB_ROWS, hub_graph

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("algo", ["weighted", "ppr", "node2vec"])
@pytest.mark.parametrize("mode", ["fast", "exact"])
def test_walks_around_the_shape_limits(algo, mode):
    need_gpu()
    built()
    from paper_2404_08364_gb300 import DeviceGraph
    n, row_ptr, col, w_f32, w_u32 = hub_graph()
    dg = DeviceGraph.from_tensors(row_ptr, col, w_f32, w_u32)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    starts = (torch.arange(40 * sms, dtype=torch.int32) % (len(HUB_ROWS) + 500)).cuda()
    kw = dict(mode=mode, p=2.0, q=0.5, ppr_stop=0.2)
    want = dg.walk(algo, starts, 7, 3, **kw)
    for per_sm in (24, 32):
        for n_q in (per_sm * sms - 1, per_sm * sms, per_sm * sms + 1):
            dg.stats_reset()
            got = dg.walk(algo, starts[:n_q].contiguous(), 7, 3, **kw)
            st = dg.stats()
            assert all(torch.equal(a, b[:n_q]) for a, b in zip(got, want))
            assert st["walks"] == n_q and st["steps"] == int((got[1] - 1).sum())
