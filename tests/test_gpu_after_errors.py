"""A refused allocation is reported by the call that asked for it, and by no
later one."""

import ctypes

import numpy as np
import pytest
import torch

import fw_inputs as fi
from gpu_common import cached_graph, device_graph

pytestmark = pytest.mark.gpu


def _huge_load():
    from paper_2404_08364_gb300 import _fw
    row_ptr, col = np.zeros(2, dtype=np.int64), np.zeros(1, dtype=np.int32)
    h = ctypes.c_void_p()
    # 2^42 entries: refused before any array is read
    return _fw.lib().fw_load_csr(ctypes.byref(h), 1, 1 << 42, row_ptr.ctypes.data_as(ctypes.c_void_p),
                                 col.ctypes.data_as(ctypes.c_void_p), None, None, None, _fw.FW_HOST_PTRS)


def _huge_server(dg):
    from paper_2404_08364_gb300 import _fw
    h = ctypes.c_void_p()
    return _fw.lib().fw_server_create(dg._h, 1, 1 << 44, 4, 5.0, ctypes.byref(h))


@pytest.mark.parametrize("what", ["load", "server"])
def test_a_walk_after_a_refused_allocation(what):
    from paper_2404_08364_gb300 import _fw, sample
    g = cached_graph("rmat", 12, 2)
    dg = device_graph(g)
    starts = fi.random_starts(g.n, 300, 5, "cuda")
    want = dg.walk("weighted", starts, 10, 9, mode="fast")
    w = torch.rand(500, device="cuda") + 1
    draws = sample("expj", w, 64, timed=False)[0]
    torch.cuda.synchronize()
    for call in (lambda: dg.walk("weighted", starts, 10, 9, mode="fast"), lambda: (sample("expj", w, 64, timed=False)[0],)):
        rc = _huge_load() if what == "load" else _huge_server(dg)
        assert rc == _fw.FW_ENOMEM
        got = call()
        ref = want if len(got) == 2 else (draws,)
        torch.cuda.synchronize()
        assert all(torch.equal(a, b) for a, b in zip(got, ref))
