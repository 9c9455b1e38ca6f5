"""Launches of different shapes from two threads: a kernel's limit on dynamic shared
memory belongs to the function, so a small launch's larger CTAs and a large
launch's smaller ones must not set it for each other."""

import threading

import pytest
import torch

from gpu_common import built, need_gpu
from test_gpu_row_edges import edge_graph

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", ["fast", "exact"])
def test_small_and_large_launches_from_two_threads(mode):
    need_gpu()
    built()
    from paper_2404_08364_gb300 import DeviceGraph
    g = edge_graph()
    t = [torch.from_numpy(x) for x in (g.row_ptr, g.col, g.w_f32, g.w_u32.view("int32"))]
    kw = dict(mode=mode, p=2.0, q=0.5)
    work = []
    for n_q in (8, 20000):
        dg = DeviceGraph.from_tensors(*t)
        starts = (torch.arange(n_q, dtype=torch.int32) % 25).cuda()
        work.append((dg, starts, dg.walk("node2vec", starts, 2, 7, **kw)))
    torch.cuda.synchronize()
    failed = []

    def run(dg, starts, ref):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                for _ in range(200):
                    got = dg.walk("node2vec", starts, 2, 7, stream=torch.cuda.current_stream(), **kw)
                torch.cuda.current_stream().synchronize()
            assert all(torch.equal(a, b) for a, b in zip(got, ref))
        except Exception as e:  # reported by the main thread
            failed.append(e)

    threads = [threading.Thread(target=run, args=w) for w in work]
    for th in threads:
        th.start()
    for th in threads:
        th.join()
    assert not failed, failed
